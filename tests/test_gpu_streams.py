"""Small beams on streams of their own run beside one another.

A window of few particles takes only the blocks that shorten it, so the
windows of several handles share the GPU; whatever blocks a window takes, its
results are the same bits.
"""
import threading
import time

import pytest

import oracle
from paper_1404_1160_gb300 import inputs
from paper_1404_1160_gb300 import pic
from tests.gpu_common import bit_equal, cfg_of

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_1160_gb300 import build

    build.build()
    torch.cuda.set_device(0)


def together(hs, steps):
    """Wall time of `steps` macro steps of every handle, each in its own thread."""
    ts = [threading.Thread(target=pic.pic_step, args=(h, steps)) for h in hs]
    t0 = time.perf_counter()
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    return time.perf_counter() - t0


@pytest.mark.parametrize("precision,n", [(0, 2000), (1, 2000), (1, 20_000)])
def test_small_beams_of_several_streams_overlap(precision, n):
    p = pic.pic_default_params(precision=precision)
    ys = [inputs.gaussian_beam(n, seed=k, r_cut=4.0) for k in range(4)]
    streams = [torch.cuda.Stream() for _ in ys]
    hs = [pic.pic_init(p, *y, stream=s) for y, s in zip(ys, streams)]
    one = [pic.pic_init(p, *y) for y in ys]
    # four beams of at most 40 blocks of half an SM each fit the GPU together (two by
    # two they would take twice as long as one)
    alone = min(together(one[:1], 5) for _ in range(4))
    four = min(together(hs, 5) for _ in range(4))
    assert four < 1.5 * alone, (four, alone)
    for h in one[1:]:
        pic.pic_step(h, 20)
    for h, o in zip(hs, one):
        R, V = pic.pic_get_particles(h)
        Ro, Vo = pic.pic_get_particles(o)
        assert bit_equal(R, Ro) and bit_equal(V, Vo)
        pic.pic_destroy(h)
        pic.pic_destroy(o)


# chunks per block, blocks per SM, threads per block: the lines of the default shapes (152 SMs)
EDGES = [(n, 256) for n in (127, 128, 129, 511, 513, 4 * 32 * 152, 4 * 32 * 152 + 1, 16 * 32 * 152, 16 * 32 * 152 + 1)] + [
    (3000, c) for c in (494, 496, 742, 744)]


@pytest.mark.parametrize("n,n_cells", EDGES)
def test_lines_between_the_default_shapes(n, n_cells):
    kw = dict(n_cells=n_cells, steps_per_turn=20, max_window_steps=60)
    R0, V0 = inputs.gaussian_beam(n, seed=n, r_cut=None)
    for precision in (0, 1):
        out = []
        for block in (0, 128):
            p = pic.pic_default_params(precision=precision, block_size=block, **kw)
            h = pic.pic_init(p, R0, V0)
            pic.pic_step(h, 1)
            out.append(pic.pic_get_particles(h))
            pic.pic_destroy(h)
        assert bit_equal(out[0][0], out[1][0]) and bit_equal(out[0][1], out[1][1])
        if precision == 0:
            ref = oracle.etd_step(cfg_of(p), R0, V0)
            assert bit_equal(out[0][0], ref.R) and bit_equal(out[0][1], ref.V)


def test_analytic_window_of_the_fp32_form_takes_no_smaller_blocks():
    # one-warp blocks share out the FP64 pipe; the binary32 window has no FP64 in
    # its loop, and they only made a step of 5000 particles 16 % longer
    R0, V0 = inputs.gaussian_beam(5000, seed=1)
    kw = dict(precision=1, field_model=pic.PIC_FIELD_DUFFING, sort_every=0)
    hs = [pic.pic_init(pic.pic_default_params(block_size=b, **kw), R0, V0) for b in (0, 128)]
    t = [[], []]
    for i in range(400):
        for k in (i & 1, 1 - (i & 1)):
            t0 = time.perf_counter()
            pic.pic_step(hs[k], 1)
            t[k].append(time.perf_counter() - t0)
    default, block128 = (sorted(x[40:])[len(x[40:]) // 2] for x in t)
    for h in hs:
        pic.pic_destroy(h)
    assert default < 1.05 * block128, (default, block128)
