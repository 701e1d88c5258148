"""The field cycle of the window kernels at the edges of its forms.

The charge words of a cycle count their own arrivals where n W leaves room,
else the cycle ends in a grid barrier; the field is built from 1 to 4 nodes
per thread in registers or from shared memory.  The charge is an exact
integer either way, so every form gives the same bits: FP64 windows equal the
oracle's, FP32 windows do not depend on the block size (128 threads take the
barrier and the shared-memory build on these meshes).
"""
import numpy as np
import pytest

import oracle
from paper_1404_1160_gb300 import inputs
from paper_1404_1160_gb300 import pic
from tests.gpu_common import bit_equal, cfg_of

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# nodes = 31 (block / 64) per node of a thread: 1024 threads cover 496, 992, 1488, 1984
EDGE_CELLS = [494, 496, 990, 992, 1486, 1488, 1982, 1984]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1404_1160_gb300 import build

    build.build()
    torch.cuda.set_device(0)


def etd(p, R0, V0, steps=1):
    h = pic.pic_init(p, R0, V0)
    pic.pic_step(h, steps)
    R, V = pic.pic_get_particles(h)
    Q = pic.pic_get_field(h, p.n_cells)[0]
    pic.pic_destroy(h)
    return R, V, Q


@pytest.mark.parametrize("n_cells", EDGE_CELLS)
def test_fp64_register_build_edges(n_cells):
    p = pic.pic_default_params(n_cells=n_cells, steps_per_turn=20, max_window_steps=60)
    R0, V0 = inputs.gaussian_beam(1500, seed=n_cells, r_cut=None)
    R, V, Q = etd(p, R0, V0)
    ref = oracle.etd_step(cfg_of(p), R0, V0)
    assert bit_equal(R, ref.R) and bit_equal(V, ref.V)
    assert np.array_equal(Q, oracle.deposit(cfg_of(p), ref.R)[0])


@pytest.mark.parametrize("n_cells", EDGE_CELLS)
def test_fp32_register_build_edges(n_cells):
    R0, V0 = inputs.gaussian_beam(1500, seed=n_cells, r_cut=None)
    kw = dict(precision=1, n_cells=n_cells, steps_per_turn=20, max_window_steps=60)
    a = etd(pic.pic_default_params(**kw), R0, V0, 2)
    b = etd(pic.pic_default_params(block_size=128, **kw), R0, V0, 2)
    assert all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("n,log2W", [(60_000, 40), (70_000, 40), (140_000, 40), (300, 32), (1, 32), (33, 40)])
def test_count_bits_of_the_charge_words(n, log2W):
    # n W on both sides of what the words hold beside the count (64 bits in all)
    p = pic.pic_default_params(weight_fixed=1 << log2W, steps_per_turn=20, max_window_steps=60)
    R0, V0 = inputs.gaussian_beam(n, seed=n, r_cut=4.0)
    R, V, Q = etd(p, R0, V0)
    ref = oracle.etd_step(cfg_of(p), R0, V0)
    assert bit_equal(R, ref.R) and bit_equal(V, ref.V)
    assert np.array_equal(Q, oracle.deposit(cfg_of(p), ref.R)[0])


def test_all_particles_on_one_node():
    # the whole charge n W in one word of every cycle (R = V = 0 stays on the axis)
    n = 200_000
    p = pic.pic_default_params(steps_per_turn=20, max_window_steps=60, field_parity=pic.PIC_PARITY_ODD)
    R, V, Q = etd(p, np.zeros(n), np.zeros(n), 2)
    assert not R.any() and not V.any()
    assert Q[p.n_cells // 2] == n * p.weight_fixed and Q.sum() == n * p.weight_fixed


# FP64 chunks of 32 particles: kept in shared memory (small n), staged one
# ahead (large n) or loaded in place (large meshes); 152 SMs
WAYS = [(1, {}), (31, {}), (33, {}), (152 * 32 - 1, {}), (152 * 32 + 1, {}), (5000, dict(block_size=512, blocks_per_sm=2)),
        (20_000, dict(n_cells=2048)), (400_000, {}), (480_000, {}), (480_000, dict(n_cells=100))]


@pytest.mark.parametrize("n,kw", WAYS)
@pytest.mark.parametrize("solver", [pic.PIC_FINE_RK4, pic.PIC_FINE_LAWSON_RK4])
def test_fp64_ways_to_keep_the_chunks(n, kw, solver):
    p = pic.pic_default_params(fine_solver=solver, steps_per_turn=20, max_window_steps=60, **kw)
    cfg = cfg_of(p)
    R0, V0 = inputs.gaussian_beam(n, seed=n, r_cut=None)
    h = pic.pic_init(p, R0, V0)
    pic.pic_step(h, 1)
    R, V = pic.pic_get_particles(h)
    T, N, o = pic.pic_get_periods(h)
    ref = oracle.etd_step(cfg, R0, V0)
    assert bit_equal(R, ref.R) and bit_equal(V, ref.V) and np.array_equal(N, ref.N)
    # the reference solution and step 1 alone (the modified scheme) on the same handle
    pic.pic_set_particles(h, R0, V0)
    pic.pic_fine_steps(h, 3)
    R, V = pic.pic_get_particles(h)
    Rf, Vf = oracle.fine_steps(cfg, R0, V0, 3)
    assert bit_equal(R, Rf) and bit_equal(V, Vf)
    pic.pic_set_particles(h, R0, V0)
    P = pic.pic_step_classic(h, 1, 1)
    R, V = pic.pic_get_particles(h)
    Rc, Vc, Pc = oracle.classic_step(cfg, R0, V0, 1)
    assert P == Pc and bit_equal(R, Rc) and bit_equal(V, Vc)
    assert bit_equal(pic.pic_get_periods(h)[2], o)  # step 1 alone leaves the last macro step's remainders
    pic.pic_destroy(h)


@pytest.mark.parametrize("n", [32, 3000, 100_000, 700_000, 2_000_000])
@pytest.mark.parametrize("n_cells", [256, 100, 1024])
def test_fp32_deposit_forms_agree(n, n_cells):
    # a warp with an off-mesh lane deposits in the general form, another one in
    # the fast form: the same particles give the same bits in both.  Every
    # second slot of run B holds a far particle (off the mesh for these few
    # steps); twice the charge keeps the charge unit.
    rng = np.random.default_rng(n + n_cells)
    R0 = rng.uniform(-3.7, 3.9, n)
    V0 = rng.normal(0, 0.5, n)
    far = np.where(np.arange(2 * n) % 2 == 0, 100.0, 0.0)
    RB, VB = far.copy(), np.zeros(2 * n)
    RB[1::2], VB[1::2] = R0, V0
    out = []
    for R, V, charge in ((R0, V0, 1.0), (RB, VB, 2.0)):
        p = pic.pic_default_params(precision=1, n_cells=n_cells, sort_every=0, total_charge=charge)
        h = pic.pic_init(p, R, V)
        pic.pic_fine_steps(h, 3)
        out.append(pic.pic_get_particles(h))
        pic.pic_destroy(h)
    (Ra, Va), (Rb, Vb) = out
    assert np.array_equal(Ra, Rb[1::2]) and np.array_equal(Va, Vb[1::2])


def test_fp32_blocks_past_the_parts_of_the_fast_split():
    # more than 2^20 positions per block and copy: the 11/11/10-bit split
    n = (1 << 20) + 4096
    rng = np.random.default_rng(3)
    R0, V0 = rng.normal(0, 1, n), rng.normal(0, 1, n)
    kw = dict(precision=1, steps_per_turn=4, max_window_steps=10, r_min=-8.0, r_max=8.0)
    a = etd(pic.pic_default_params(**kw), R0, V0)
    params = [pic.pic_default_params(**kw)]
    b = pic.pic_batch_create(params + [pic.pic_default_params(precision=1, field_model=pic.PIC_FIELD_ZERO)] * 151,
                             [(R0, V0)] + [(np.ones(1), np.ones(1))] * 151)
    pic.pic_batch_step(b, 1)  # 152 beams on 152 blocks: the large one has a single block
    R, V = pic.pic_batch_get_particles(b, 0)
    b.close()
    assert np.array_equal(R, a[0]) and np.array_equal(V, a[1])
