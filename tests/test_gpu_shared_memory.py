"""The shared memory that a launch may take belongs to the kernel, which all
handles and batches of a process share: no handle may take it from another,
and every mesh that the windows serve has to launch.
"""
import ctypes as C
import threading

import numpy as np
import pytest

import oracle
from oracle import learned as OL
from oracle import mlp as omlp
from paper_1404_1160_gb300 import inputs
from paper_1404_1160_gb300 import pic
from tests.gpu_common import bit_equal, cfg_of
from tests.test_gpu_f32 import f32

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHORT = dict(steps_per_turn=20, max_window_steps=60)


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_1160_gb300 import build

    build.build()
    torch.cuda.set_device(0)


# (particles, cells) of handles that live at the same time, the one that takes
# the most shared memory first
TOGETHER = [[(20_000, 256), (2000, 256)], [(2000, 1024), (2000, 256)], [(400_000, 256), (3000, 128), (3000, 2048)]]


@pytest.mark.parametrize("sizes", TOGETHER)
@pytest.mark.parametrize("solver", [pic.PIC_FINE_RK4, pic.PIC_FINE_LAWSON_RK4])
def test_fp64_handles_step_in_turn(sizes, solver):
    runs = []
    for n, cells in sizes:
        p = pic.pic_default_params(n_cells=cells, fine_solver=solver, **SHORT)
        y = inputs.gaussian_beam(n, seed=n, r_cut=4.0)
        runs.append([p, y, pic.pic_init(p, *y)])
    for _ in range(2):
        for r in runs:
            pic.pic_step(r[2], 1)
            ref = oracle.etd_step(cfg_of(r[0]), *r[1])
            R, V = pic.pic_get_particles(r[2])
            assert bit_equal(R, ref.R) and bit_equal(V, ref.V)
            r[1] = (ref.R, ref.V)
    for r in runs:
        pic.pic_destroy(r[2])


def alone(p, y, steps):
    h = pic.pic_init(p, *y)
    pic.pic_step(h, steps)
    out = pic.pic_get_particles(h)
    pic.pic_destroy(h)
    return out


@pytest.mark.parametrize("sizes", TOGETHER + [[(700_000, 512), (650_000, 100)]])
def test_fp32_handles_step_in_turn(sizes):
    ps = [pic.pic_default_params(precision=1, n_cells=cells, **SHORT) for _, cells in sizes]
    ys = [inputs.gaussian_beam(n, seed=n, r_cut=4.0) for n, _ in sizes]
    ref = [alone(p, y, 2) for p, y in zip(ps, ys)]
    hs = [pic.pic_init(p, *y) for p, y in zip(ps, ys)]
    for _ in range(2):
        for h in hs:
            pic.pic_step(h, 1)
    for h, (R0, V0) in zip(hs, ref):
        R, V = pic.pic_get_particles(h)
        pic.pic_destroy(h)
        assert bit_equal(R, R0) and bit_equal(V, V0)


# 1752 cells with two histogram copies: within 1 KB of all the shared memory a block can have
@pytest.mark.parametrize("cells,copies", [(2048, 1), (1752, 2), (1752, 1)])
def test_batches_step_in_turn(cells, copies):
    specs = [[(cells, 3000), (128, 2000)], [(128, 4000), (256, 1000)]]
    bs, ref = [], []
    for k, spec in enumerate(specs):
        ps = [pic.pic_default_params(precision=1, n_cells=c, **SHORT) for c, _ in spec]
        ys = [inputs.gaussian_beam(n, seed=n, r_cut=4.0) for _, n in spec]
        ref.append([alone(p, y, 2) for p, y in zip(ps, ys)])
        bs.append(pic.pic_batch_create(ps, ys))
        if k == 0:
            pic.pic_batch_set_config(bs[0], 1024, 1, 0.85, 1, copies)
    for _ in range(2):
        for b in bs:
            pic.pic_batch_step(b, 1)
    for b, rs in zip(bs, ref):
        for i, (R0, V0) in enumerate(rs):
            R, V = pic.pic_batch_get_particles(b, i)
            assert bit_equal(R, R0) and bit_equal(V, V0)
        b.close()


@pytest.mark.parametrize("cells", [1278, 1280, 1620, 1622, 2048])
def test_learned_step_of_the_fp32_form_on_fine_meshes(cells):
    # a constant correction (W3 = 0: the output is b3 exactly) judged by the
    # frozen-field energy, with the tables of the check in shared memory
    n, scale, tol = 20_001, (2.0**-9, 2.0**-10), 2e-3
    p = pic.pic_default_params(precision=1, dt=0.4, n_cells=cells, r_min=-2.0, r_max=2.0)
    c = cfg_of(p)
    R0, V0 = (f32(x).astype(np.float64) for x in inputs.gaussian_beam(n, seed=21))
    w = np.zeros(omlp.N_PARAMS, np.float32)
    w[-2:] = (1.0, -0.75)
    m = pic.pic_mlp_create(16)
    pic.pic_mlp_set_weights(m, w)
    Rp, Vp = alone(p, (R0, V0), 1)
    h = pic.pic_init(p, R0, V0)
    n_fb = pic.pic_step_learned(h, m, 1, scale=scale, drift_tol=tol)
    R, V = pic.pic_get_particles(h)
    assert pic.pic_moments(h)["n_steps"] == 1
    pic.pic_destroy(h)
    m.close()
    E, edges = OL.mesh_field(c, R0, n, precision=1)
    Ro, Vo, keep, margin = OL.learned_apply(c, Rp, Vp, np.full(n, scale[0]), np.full(n, -0.75 * scale[1]), tol, E, edges, 1)
    # the decision is the oracle's but within the rounding of H on either side
    psi = float(np.abs(OL.node_potential(c, E)).max())
    sure = np.abs(margin) > 1e-10 * (np.abs(OL.frozen_energy(c, Rp, Vp, E, edges)) + c.eps * psi)
    assert sure.mean() > 0.999 and 0.05 < keep.mean() < 0.95
    assert bit_equal(R[sure], Ro[sure]) and bit_equal(V[sure], Vo[sure])
    fb = int((~keep & sure).sum())
    assert fb <= n_fb <= fb + int((~sure).sum())


def test_mesh_calls_of_several_threads():
    # threads on meshes whose tables need different sizes above 48 KB, on their own streams and buffers
    cells = [4098, 6000, 8190]
    bad = []

    def work(c):
        p = pic.pic_default_params(n_cells=c)
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            R = torch.randn(500, dtype=torch.float64, device="cuda")
            Q = torch.empty(c + 1, dtype=torch.int64, device="cuda")
            n_out = torch.empty(1, dtype=torch.int64, device="cuda")
        s.synchronize()
        call = pic.load().pic_deposit
        args = (C.byref(p), R.numel(), R.data_ptr(), Q.data_ptr(), n_out.data_ptr(), s.cuda_stream)
        status = [call(*args) for _ in range(10_000)]
        s.synchronize()
        Qo, no = oracle.deposit(cfg_of(p), R.cpu().numpy())
        if any(status) or not np.array_equal(Q.cpu().numpy(), Qo) or int(n_out) != no:
            bad.append((c, sum(x != 0 for x in status)))

    threads = [threading.Thread(target=work, args=(c,)) for c in cells]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
