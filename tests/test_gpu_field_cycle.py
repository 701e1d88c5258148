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


# ------------------------------------------------- standalone mesh operations


@pytest.mark.parametrize("n", [1, 1023, 1025, 4097, 152 * 1024 - 1, 700_001])
@pytest.mark.parametrize("n_cells,log2W", [(2, 32), (100, 32), (1024, 32), (1026, 24), (4094, 32), (8192, 32), (8194, 32), (256, 40)])
def test_deposit_forms(n, n_cells, log2W):
    p = pic.pic_default_params(n_cells=n_cells, weight_fixed=1 << log2W)
    rng = np.random.default_rng(n + n_cells)
    R = rng.normal(0, 2, n)
    R[rng.random(n) < 0.3] = 0.01  # many positions in one cell
    R[:: max(1, n // 7)] = [np.nan, -4.0, 4.0, np.inf, -np.inf, 3.9999999, -0.0][: len(R[:: max(1, n // 7)])] if n < 7 else np.resize(
        [np.nan, -4.0, 4.0, np.inf, -np.inf, 3.9999999, -0.0], len(R[:: max(1, n // 7)]))
    Q = torch.full((n_cells + 1,), 5, dtype=torch.int64, device="cuda")
    n_out = torch.full((1,), 5, dtype=torch.int64, device="cuda")
    pic.pic_deposit(p, torch.from_numpy(R).cuda(), Q, n_out)
    Qo, no = oracle.deposit(cfg_of(p), R)
    assert np.array_equal(Q.cpu().numpy(), Qo) and int(n_out) == no
    Rf = R.astype(np.float32)
    pic.pic_deposit_f32(p, torch.from_numpy(Rf).cuda(), Q, n_out)
    Qo, no = oracle.deposit_f32(cfg_of(p), Rf)
    assert np.array_equal(Q.cpu().numpy(), Qo) and int(n_out) == no


@pytest.mark.parametrize("n_cells", [2, 30, 510, 512, 514, 1022, 1024, 2046, 2048, 4094, 4096, 8192, 16382, 16384])
@pytest.mark.parametrize("parity", [pic.PIC_PARITY_EVEN, pic.PIC_PARITY_ODD])
def test_field_from_one_block(n_cells, parity):
    p = pic.pic_default_params(n_cells=n_cells, field_parity=parity)
    Q = np.random.default_rng(n_cells).integers(0, 1 << 40, n_cells + 1).astype(np.int64)
    E = torch.empty(n_cells + 1, dtype=torch.float64, device="cuda")
    edges = torch.empty(2, dtype=torch.float64, device="cuda")
    pic.pic_poisson(p, 12345, torch.from_numpy(Q).cuda(), E, edges)
    _, Eo, eo = oracle.poisson(cfg_of(p), Q, 12345)
    assert bit_equal(E.cpu().numpy(), Eo) and bit_equal(edges.cpu().numpy(), eo)


@pytest.mark.parametrize("n_cells", [256, 1024, 4094, 8192, 16382, 16384])
def test_field_in_the_storage_of_the_charge(n_cells):
    p = pic.pic_default_params(n_cells=n_cells)
    Q = np.random.default_rng(n_cells).integers(0, 1 << 40, n_cells + 1).astype(np.int64)
    q = torch.from_numpy(Q).cuda()
    edges = torch.empty(2, dtype=torch.float64, device="cuda")
    pic.pic_poisson(p, 12345, q, q.view(torch.float64), edges)
    _, Eo, eo = oracle.poisson(cfg_of(p), Q, 12345)
    assert bit_equal(q.view(torch.float64).cpu().numpy(), Eo) and bit_equal(edges.cpu().numpy(), eo)


@pytest.mark.parametrize("n_cells", [2, 6, 512, 1022, 1026, 65536])
def test_frozen_potential_of_any_mesh(n_cells):
    # psi at the nodes against long double sums: (n_cells + 4) binary64 roundings of
    # the largest partial sum bound the run and scan sums of either side
    p = pic.pic_default_params(n_cells=n_cells)
    E = np.random.default_rng(n_cells).normal(0, 1, n_cells + 1)
    hr, c = 8.0 / n_cells, n_cells // 2
    inc = np.longdouble(0.5 * hr) * (E[:-1].astype(np.longdouble) + E[1:])
    ref = np.concatenate([-np.cumsum(inc[:c][::-1])[::-1], [0], np.cumsum(inc[c:])])
    psi = torch.empty(n_cells + 1, dtype=torch.float64, device="cuda")
    out = torch.empty(1, dtype=torch.float64, device="cuda")
    pic.pic_frozen_potential(p, torch.from_numpy(E).cuda(), torch.zeros(2, dtype=torch.float64, device="cuda"), psi,
                             torch.zeros(1, dtype=torch.float64, device="cuda"), out)
    bound = (n_cells + 4) * 2.0**-53 * float(np.sum(np.abs(inc)))
    assert np.max(np.abs(psi.cpu().numpy() - ref.astype(np.float64))) <= bound


# without a field table in shared memory (more than 6144 cells): one position per thread in flight, or
# four beyond 36 per thread of four blocks on each of 152 SMs
@pytest.mark.parametrize("n", [1, 255, 257, 4 * 256 * 152 + 1, 36 * 4 * 256 * 152, 36 * 4 * 256 * 152 + 1])
@pytest.mark.parametrize("n_cells,r_max", [(6146, 4.0), (65536, 8.0)])
def test_gather_without_a_table(n, n_cells, r_max):
    p = pic.pic_default_params(n_cells=n_cells, r_min=-r_max, r_max=r_max)
    rng = np.random.default_rng(n)
    R, E, edges = rng.normal(0, 0.5 * r_max, n), rng.normal(0, 1, n_cells + 1), rng.normal(0, 1, 2)
    R[: min(n, 5)] = [r_max, -r_max, 0.0, np.nan, -np.inf][: min(n, 5)]
    e = torch.empty(n, dtype=torch.float64, device="cuda")
    pic.pic_gather(p, torch.from_numpy(R).cuda(), torch.from_numpy(E).cuda(), torch.from_numpy(edges).cuda(), e)
    eo = oracle.gather(cfg_of(p), R, E, edges)
    nan = np.isnan(eo)
    assert np.array_equal(nan, np.isnan(e.cpu().numpy())) and bit_equal(e.cpu().numpy()[~nan], eo[~nan])
