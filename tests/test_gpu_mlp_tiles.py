"""The network's kernels at the edges of their 128-sample tiles and of the
tiles per block (152 SMs): forward and gradients inside the oracle's binary32
intervals, as in tests/test_gpu_mlp.py."""
import numpy as np
import pytest

from oracle import mlp as omlp
from paper_1404_1160_gb300 import pic
from tests.test_gpu_mlp import batch, dev, weights

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_1160_gb300 import build

    build.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("n", [1, 127, 128, 129, 152 * 128 + 5, 3 * 152 * 128 - 1])
def test_gradients_at_tile_edges(n):
    m = pic.pic_mlp_create(n)
    w = weights(5)
    pic.pic_mlp_set_weights(m, w)
    X, T = batch(n, n)
    g, loss = pic.pic_mlp_gradients(m, dev(X), dev(T))
    # longest chain of sequential additions: 16 samples of each of a block's
    # tiles per thread, the 8 threads of a unit, then the blocks
    tiles = -(-n // 128)
    blocks = min(tiles, 152)
    n_seq = 16 * -(-tiles // blocks) + 8 + blocks + 2
    loss_iv, g_iv = omlp.grads_interval(w.astype(np.float64), X.astype(np.float64), T.astype(np.float64), n_seq)
    assert loss_iv.lo <= loss <= loss_iv.hi
    outside = (g < g_iv.lo) | (g > g_iv.hi)
    assert not outside.any(), (np.argwhere(outside)[:5].ravel(), g[outside][:5], g_iv.mid[outside][:5])
    m.close()


@pytest.mark.parametrize("block", [(name, at) for name in ("W1", "b1", "W2", "b2", "W3", "b3") for at in (0, -1)])
def test_rows_past_the_batch_add_nothing(block):
    # one sample repeated: 127 rows and a whole tile of 128 have the same infinities
    # and NaNs in every gradient, also where a weight is infinite
    p = omlp.unflatten(weights(8).astype(np.float64))
    p[block[0]].flat[block[1]] = np.inf
    w = omlp.flatten(p).astype(np.float32)
    X, T = batch(1, 4)
    out = []
    for n in (127, 128):
        m = pic.pic_mlp_create(n)
        pic.pic_mlp_set_weights(m, w)
        out.append(pic.pic_mlp_gradients(m, dev(np.repeat(X, n, 0)), dev(np.repeat(T, n, 0)))[0])
        m.close()
    assert np.array_equal(np.isnan(out[0]), np.isnan(out[1]))
    assert np.array_equal(np.isposinf(out[0]), np.isposinf(out[1])) and np.array_equal(np.isneginf(out[0]), np.isneginf(out[1]))


@pytest.mark.parametrize("n", [127, 129, 12 * 152 * 128 + 1])
def test_forward_at_tile_edges(n):
    m = pic.pic_mlp_create(16)
    w = weights(6)
    pic.pic_mlp_set_weights(m, w)
    X, _ = batch(n, n)
    Y = torch.full((n, 2), float("nan"), dtype=torch.float32, device="cuda")
    pic.pic_mlp_forward(m, dev(X), Y)
    iv = omlp.forward_interval(w.astype(np.float64), X.astype(np.float64))["out"]
    y = Y.cpu().numpy().astype(np.float64)
    assert ((y >= iv.lo) & (y <= iv.hi)).all()
    m.close()


def test_losses_of_a_long_training():
    # the losses are copied to the host in runs; a longer training repeats a shorter one's
    X, T = batch(500, 9)
    hist = []
    for steps in (10, 4096, 4100):
        m = pic.pic_mlp_create(64)
        pic.pic_mlp_set_weights(m, weights(7))
        hist.append(pic.pic_mlp_train(m, dev(X), dev(T), batch=64, steps=steps, lr=1e-4, seed=3))
        m.close()
    assert all(h.size == k and np.isfinite(h).all() for h, k in zip(hist, (10, 4096, 4100)))
    assert np.array_equal(hist[0], hist[2][:10]) and np.array_equal(hist[1], hist[2][:4096])
    assert len(np.unique(hist[2][4090:])) == 10
