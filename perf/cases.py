"""The work that programs have this library do, as cases that can be timed.

A case is a dict of plain values.  Its "kind" says which calls a pass makes:

  step      a program that owns (R, V): pic_set_particles, macro steps of one
            scheme, pic_get_particles
  learned   the same around pic_step_learned
  batch     the same for many beams in one launch (pic_batch_*)
  mesh      one field cycle on the caller's own buffers: deposit, field, gather
  diag      the diagnostics of a running beam: moments, field, periods
  forward   the network of the learned stepper on many samples
  train     Adam steps of that network on batches of a data set

Every array a pass needs is on the GPU before it starts; a pass returns the
arrays the calls filled.  exact() computes the same results in FP64 with
plain torch operations.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1404_1160_gb300 import inputs
from paper_1404_1160_gb300 import pic

PAPER = dict(beam="paper", r_max=2.0, n_cells=256, eps=1e-3, dt=0.5)
GAUSS = dict(beam="gauss", r_max=4.0, n_cells=256, eps=1e-2, dt=0.1)
STEP = dict(kind="step", precision=0, field="poisson", solver="lawson", scheme="etd", cap=300, once=False, sort=4, steps=1)


def listed():
    return [
        # the paper's own Vlasov-Poisson run (Sec. 4.2): 20000 particles, explicit RK4, a few steps between outputs
        dict(STEP, **PAPER, name="paper_2e4", n=20000, solver="rk4", sort=1, steps=2),
        # the benchmark beam
        dict(STEP, **GAUSS, name="beam_1e6", n=10**6),
        # the comparator scheme between the sizes, on a mesh whose spacing is no power of two
        dict(STEP, **dict(GAUSS, n_cells=100), name="modified_1.5e5", n=150001, scheme="modified", sort=1),
        # the Duffing test run: periods known from the start, 20 steps between outputs
        dict(STEP, **dict(GAUSS, beam="wide", dt=0.05), name="duffing_1e4", n=10000, field="duffing", once=True, sort=0, steps=20),
        # the binary32 form on the benchmark beam, and on a large one
        dict(STEP, **GAUSS, name="beam32_1e6", n=10**6, precision=1),
        dict(STEP, **dict(GAUSS, n_cells=1024, eps=1e-3), name="beam32_2e7", n=20_000_003, precision=1, cap=202),
        # large steps with the network's correction
        dict(STEP, **dict(GAUSS, n_cells=512, dt=0.4), name="learned32_2e6", kind="learned", n=2 * 10**6, precision=1, tol=1e-4),
        # many uneven beams at once
        dict(kind="batch", name="batch_12", beams=12, log_lo=4.0, log_hi=5.7, dt=0.1),
        # a field cycle on a program's own positions
        dict(kind="mesh", name="mesh_1e6", n=1_000_003, n_cells=256, r_max=4.0, precision=0),
        # what a run prints after a step
        dict(STEP, **GAUSS, name="diag_1e6", kind="diag", n=10**6),
        # the network: inference on a ragged set, training at its usual batch
        dict(kind="forward", name="forward_1e5", n=100_003),
        dict(kind="train", name="train_8192", n=300_000, batch=8192, steps=5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step32", "step32", "duffing", "learned", "batch", "mesh", "mesh", "diag", "forward", "train"])
    cells = rng.choice([100, 128, 256, 256, 512, 1000, 1024])
    eps, dt = rng.choice([0.05, 0.01, 0.005, 0.001]), rng.choice([0.1, 0.2, 0.4, 0.5])
    gauss = dict(GAUSS, n_cells=cells, eps=eps, dt=dt)
    sort = rng.choice([1, 4])
    if kind == "step":
        beam = dict(PAPER) if rng.random() < 0.25 else gauss
        return dict(STEP, **beam, n=_log_int(rng, 2e3, 1e6), solver=rng.choice(["lawson", "rk4"]), sort=sort,
                    scheme=rng.choice(["etd", "etd", "classic", "modified", "fine"]))
    if kind == "step32":
        return dict(STEP, **gauss, n=_log_int(rng, 2e4, 1e7), precision=1, cap=rng.choice([202, 300]), sort=sort)
    if kind == "duffing":
        return dict(STEP, **dict(GAUSS, beam="wide", eps=eps, dt=rng.choice([0.05, 0.1, 0.5])), n=_log_int(rng, 1e3, 5e5), field="duffing",
                    once=rng.random() < 0.5, sort=0, steps=rng.choice([1, 5, 20]), precision=rng.choice([0, 1]))
    if kind == "learned":
        return dict(STEP, **dict(gauss, dt=0.4, eps=0.01), kind="learned", n=_log_int(rng, 2e4, 2e6), precision=rng.choice([0, 1, 1]), sort=sort, tol=1e-4)
    if kind == "batch":
        return dict(kind="batch", beams=rng.randint(4, 16), log_lo=4.0, log_hi=rng.choice([5.0, 5.3, 5.7]), dt=0.1)
    if kind == "mesh":
        return dict(kind="mesh", n=_log_int(rng, 1e3, 2e7), n_cells=rng.choice([64, 100, 256, 512, 1024, 4096, 10000, 65536]), r_max=4.0,
                    precision=rng.choice([0, 1]))
    if kind == "diag":
        return dict(STEP, **gauss, kind="diag", n=_log_int(rng, 2e4, 2e6), precision=rng.choice([0, 1]), sort=sort)
    if kind == "forward":
        return dict(kind="forward", n=_log_int(rng, 1e2, 1e7))
    return dict(kind="train", n=_log_int(rng, 2e4, 1e6), batch=rng.choice([1000, 2048, 4096, 8192, 16384]), steps=rng.randint(2, 8))


# ------------------------------------------------------------ inputs


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _beam(beam, n, seed, precision=0):
    """(R, V) on the GPU, FP64 (rounded to binary32 values for the binary32 form)."""
    g = _gen(seed)
    u = torch.rand(n, dtype=torch.float64, device="cuda", generator=g) * 2 - 1
    v = torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
    if beam == "paper":
        r, v = inputs.PAPER_R_HALF_WIDTH * u, inputs.PAPER_V_TH * v
    elif beam == "gauss":  # N(0, 1) cut at |r| = 4
        r = math.sqrt(2.0) * torch.erfinv(u * math.erf(4.0 / math.sqrt(2.0)))
    else:
        r = math.sqrt(2.0) * torch.erfinv(u.clamp(-1 + 1e-9, 1 - 1e-9))
    return (r.float().double(), v.float().double()) if precision else (r, v)


def _params(c):
    return pic.pic_default_params(
        eps=c["eps"], dt=c["dt"], n_cells=c["n_cells"], r_min=-c["r_max"], r_max=c["r_max"], precision=c["precision"],
        field_model=pic.PIC_FIELD_POISSON if c["field"] == "poisson" else pic.PIC_FIELD_DUFFING,
        fine_solver=pic.PIC_FINE_RK4 if c["solver"] == "rk4" else pic.PIC_FINE_LAWSON_RK4,
        max_window_steps=c["cap"], periods_once=int(c["once"]), sort_every=c["sort"])


def _batch_cases(c, seed):
    """One step case per beam: sizes spread over their logarithm, meshes, eps and fields in turn."""
    out = []
    for i in range(c["beams"]):
        n = int(round(10 ** (c["log_lo"] + (c["log_hi"] - c["log_lo"]) * ((i * 0.6180339887 + 0.35) % 1.0)))) + i
        b = dict(STEP, **dict(GAUSS, dt=c["dt"], eps=(0.1, 0.05, 0.01, 0.005, 0.001)[i % 5], n_cells=(128, 256, 512, 1024)[i % 4]), n=n, precision=1)
        if i % 6 == 5:
            b.update(field="duffing", once=True, beam="wide", n=min(n, 100_000 + i))
        out.append(b)
    return out


def _samples(n, seed, dt=0.4):
    """Network inputs and targets as a run gives them: (R, V, sin, cos, dt) and a smooth correction of unit size with noise."""
    r, v = _beam("gauss", n, seed)
    g = _gen(seed + 7919)
    ph = torch.rand(n, dtype=torch.float64, device="cuda", generator=g) * (2 * math.pi)
    X = torch.stack([r, v, ph.sin(), ph.cos(), torch.full_like(r, dt)], dim=1).float()
    noise = 0.1 * torch.randn(n, 2, dtype=torch.float64, device="cuda", generator=g)
    T = (torch.stack([torch.sin(r) * ph.cos(), torch.tanh(v) * r * 0.5], dim=1) + noise).float()
    return X.contiguous(), T.contiguous()


def _scale():
    return 2e-5, 1e-5  # what the corrections of a Delta t = 0.4 step come to


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"case": c}
    if kind in ("step", "learned", "diag"):
        s["r0"], s["v0"] = _beam(c["beam"], c["n"], seed, c["precision"])
        s["h"] = pic.pic_init(_params(c), s["r0"], s["v0"])
        s["r"], s["v"] = torch.empty_like(s["r0"]), torch.empty_like(s["v0"])
        if kind == "learned":
            s["net"] = pic.pic_mlp_create(1024)
            pic.pic_mlp_set_weights(s["net"], inputs.mlp_init(seed))
        if kind == "diag":
            pic.pic_step(s["h"], 1)
    elif kind == "batch":
        s["beams"] = _batch_cases(c, seed)
        s["y0"] = [_beam(b["beam"], b["n"], seed + i, 1) for i, b in enumerate(s["beams"])]
        s["b"] = pic.pic_batch_create([_params(b) for b in s["beams"]], [(r.cpu().numpy(), v.cpu().numpy()) for r, v in s["y0"]])
        s["y"] = [(torch.empty_like(r), torch.empty_like(v)) for r, v in s["y0"]]
    elif kind == "mesh":
        s["p"] = pic.pic_default_params(n_cells=c["n_cells"], r_min=-c["r_max"], r_max=c["r_max"], precision=0)
        s["R"] = _beam("wide", c["n"], seed, c["precision"])[0]
        s["Rd"] = s["R"].float() if c["precision"] else s["R"]
        s["Q"] = torch.empty(c["n_cells"] + 1, dtype=torch.int64, device="cuda")
        s["n_out"] = torch.empty(1, dtype=torch.int64, device="cuda")
        s["E"] = torch.empty(c["n_cells"] + 1, dtype=torch.float64, device="cuda")
        s["edges"] = torch.empty(2, dtype=torch.float64, device="cuda")
        s["e"] = torch.empty(c["n"], dtype=torch.float64, device="cuda")
    elif kind == "forward":
        s["X"], _ = _samples(c["n"], seed)
        s["net"] = pic.pic_mlp_create(1024)
        pic.pic_mlp_set_weights(s["net"], inputs.mlp_init(seed))
        s["Y"] = torch.empty(c["n"], 2, dtype=torch.float32, device="cuda")
    else:
        s["X"], s["T"] = _samples(c["n"], seed)
        s["net"] = pic.pic_mlp_create(min(c["batch"], c["n"]))
        s["w0"] = inputs.mlp_init(seed)
    return s


def _scheme(h, c):
    if c["scheme"] == "etd":
        pic.pic_step(h, c["steps"])
    elif c["scheme"] == "fine":  # the paper's reference solution over one turn
        pic.pic_fine_advance(h, 2 * math.pi * c["eps"] * 1.005)
    else:
        return pic.pic_step_classic(h, c["steps"], 1 if c["scheme"] == "modified" else 0)
    return None


def run(state):
    s, c, kind = state, state["case"], state["case"]["kind"]
    if kind in ("step", "learned"):
        pic.pic_set_particles(s["h"], s["r0"], s["v0"])
        if kind == "learned":
            more = pic.pic_step_learned(s["h"], s["net"], c["steps"], scale=_scale(), drift_tol=c["tol"])
        else:
            more = _scheme(s["h"], c)
        pic.pic_get_particles(s["h"], s["r"], s["v"])
        return {"r": s["r"], "v": s["v"], "more": more}
    if kind == "batch":
        for i, (r, v) in enumerate(s["y0"]):
            pic.pic_batch_set_particles(s["b"], i, r, v)
        pic.pic_batch_step(s["b"], 1)
        for i, (r, v) in enumerate(s["y"]):
            pic.pic_batch_get_particles_into(s["b"], i, r, v)
        return s["y"]
    if kind == "mesh":
        (pic.pic_deposit_f32 if c["precision"] else pic.pic_deposit)(s["p"], s["Rd"], s["Q"], s["n_out"])
        pic.pic_poisson(s["p"], c["n"], s["Q"], s["E"], s["edges"])
        pic.pic_gather(s["p"], s["R"], s["E"], s["edges"], s["e"])
        return {"Q": s["Q"], "n_out": s["n_out"], "E": s["E"], "edges": s["edges"], "e": s["e"]}
    if kind == "diag":
        m = pic.pic_moments(s["h"])
        Q, E, edges, n_out = pic.pic_get_field(s["h"], c["n_cells"])
        T, N, o = pic.pic_get_periods(s["h"])
        # the window's time is no result, and t, the step counts and replays say how often the state was stepped
        m = {k: m[k] for k in ("n_particles", "Q_total", "n_out_of_mesh", "charge", "kinetic", "mean_R", "mean_V", "rms_R", "rms_V", "T_min",
                               "T_mean", "T_max", "N_min", "N_max", "n_no_period")}
        return {"m": m, "Q": Q, "E": E, "edges": edges, "n_out": n_out, "T": T, "N": N, "o": o}
    if kind == "forward":
        pic.pic_mlp_forward(s["net"], s["X"], s["Y"])
        return s["Y"]
    pic.pic_mlp_set_weights(s["net"], s["w0"])
    hist = pic.pic_mlp_train(s["net"], s["X"], s["T"], batch=min(c["batch"], c["n"]), steps=c["steps"], seed=0)
    grad, loss = pic.pic_mlp_gradients(s["net"], s["X"][: min(c["batch"], c["n"])], s["T"][: min(c["batch"], c["n"])])
    return {"w": pic.pic_mlp_get_weights(s["net"]), "hist": hist, "grad": grad, "loss": loss}


# ------------------------------------------------------------ work

_MLP_FLOPS = 2 * (64 * 5 + 64 * 64 + 2 * 64)


def _fine_steps(c):
    """Fine steps that one macro step cannot do without (100 per turn): the first tour of the last particle, 1.5 turns at most, and
    the window up to the landing at o + T."""
    D = c["dt"] / (2 * math.pi * c["eps"] / 100)
    if c["scheme"] == "fine":
        return 101
    if c["scheme"] != "etd":
        return 100 + D % 100 + (150 if c["scheme"] == "modified" and not c["once"] else 0)
    land = D % 100 + (100 if D >= 100 else 0) + 2
    return land if c["once"] else max(152, land)


def work(case):
    c, kind = case, case["kind"]
    if kind in ("step", "learned"):
        # 56 operations a particle and fine step with the mesh field, 34 with the analytic one; the state once in and out
        per = 56 if c["field"] == "poisson" else 34
        f = c["n"] * _fine_steps(c) * per * c["steps"] + (c["n"] * _MLP_FLOPS if kind == "learned" else 0)
        return {"bytes": 32.0 * c["n"], "flops": float(f)}
    if kind == "batch":
        each = [work(b) for b in _batch_cases(c, 0)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    if kind == "mesh":
        return {"bytes": (20.0 if c["precision"] else 16.0) * c["n"] + 16.0 * c["n_cells"], "flops": 12.0 * c["n"]}
    if kind == "diag":
        # state, T, o, N and flags in; T, N, o out
        return {"bytes": ((8 + 8 + 8 + 4 + 4) if c["precision"] else (16 + 8 + 8 + 4 + 4)) * c["n"] + 24.0 * c["n"], "flops": 20.0 * c["n"]}
    if kind == "forward":
        return {"bytes": 28.0 * c["n"], "flops": float(_MLP_FLOPS * c["n"])}
    b = min(c["batch"], c["n"])
    return {"bytes": 28.0 * b * (c["steps"] + 1), "flops": 3.0 * _MLP_FLOPS * b * (c["steps"] + 1)}


# ------------------------------------------------------------ the same in 64 bits


class _Beam:
    """Fine solver, field and macro steps of one beam in FP64 torch."""

    def __init__(self, c):
        self.c, self.eps, self.spt = c, c["eps"], 100
        self.h = 2 * math.pi * c["eps"] / self.spt
        self.nc, self.hr, self.rm = c["n_cells"], 2 * c["r_max"] / c["n_cells"], -c["r_max"]
        self.poisson = c["field"] == "poisson"
        self.nodes = self.rm + self.hr * torch.arange(self.nc + 1, dtype=torch.float64, device="cuda")

    def locate(self, R):
        x = (R - self.rm) / self.hr
        inside = (x >= 0) & (x < self.nc)
        j = torch.where(inside, x, torch.zeros_like(x)).floor()
        return inside, j.long(), torch.where(inside, x - j, torch.zeros_like(x)), x < 0

    def charge(self, R):
        inside, j, f, _ = self.locate(R)
        w = inside.double()
        return torch.bincount(j, (1 - f) * w, self.nc + 1) + torch.bincount(j + 1, f * w, self.nc + 1)

    def node_field(self, q, n):
        q, k = q / n, self.nc // 2  # total charge 1
        S = torch.cat([torch.zeros(1, dtype=torch.float64, device="cuda"), (0.5 * (q[1:] + q[:-1])).cumsum(0)])
        S = S - S[k]
        E = S / self.nodes
        E[k] = q[k] / self.hr
        return E, torch.stack([S[0], S[-1]])

    def at(self, E, edges, R):
        inside, j, f, below = self.locate(R)
        return torch.where(inside, E[j] * (1 - f) + E[j + 1] * f, torch.where(below, edges[0], edges[1]) / R)

    def E(self, R):
        if not self.poisson:
            return -R * R * R
        return self.at(*self.node_field(self.charge(R), R.numel()), R)

    def fine(self, R, V, h):
        if self.c["solver"] == "rk4":
            def f(r, v):
                return v / self.eps, -r / self.eps + self.E(r)
            a = f(R, V)
            b = f(R + 0.5 * h * a[0], V + 0.5 * h * a[1])
            c = f(R + 0.5 * h * b[0], V + 0.5 * h * b[1])
            d = f(R + h * c[0], V + h * c[1])
            return tuple(y + h / 6 * (k1 + 2 * k2 + 2 * k3 + k4) for y, k1, k2, k3, k4 in zip((R, V), a, b, c, d))
        t = h / self.eps
        c, s, ch, sh = math.cos(t), math.sin(t), math.cos(t / 2), math.sin(t / 2)
        e1 = self.E(R)
        e2 = self.E(ch * R + sh * (V + 0.5 * h * e1))
        e3 = self.E(ch * R + sh * V)
        e4 = self.E(c * R + s * V + h * sh * e3)
        return (c * R + s * V + h / 6 * (s * e1 + 2 * sh * (e2 + e3)), c * V - s * R + h / 6 * (c * e1 + 2 * ch * (e2 + e3) + e4))

    def advance(self, R, V, t):
        full = int(math.floor(t / self.h))
        for _ in range(full):
            R, V = self.fine(R, V, self.h)
        rest = t - full * self.h
        return self.fine(R, V, rest) if rest > 0 else (R, V)

    @staticmethod
    def root(v0, v1, v2):
        b, c = ((-3 * v0 + 4 * v1) - v2) / 2, ((v0 - 2 * v1) + v2) / 2
        q = -0.5 * (b + torch.where(b >= 0, 1.0, -1.0) * (b * b - 4 * v0 * c).clamp(min=0).sqrt())
        s = v0 / q
        s = torch.where((s >= 0) & (s <= 1), s, q / c)
        s = torch.where(c == 0, -v0 / b, s)
        return torch.nan_to_num(s, nan=0.0).clamp(0, 1)

    def window(self, R, V, T=None, detect=False):
        """Samples of the window and the periods; with T given, only as far as its landings need."""
        D, cap, spt = self.c["dt"] / self.h, self.c["cap"], float(self.spt)

        def decompose(T):
            T = torch.where((T > 0) & torch.isfinite(T), T, torch.full_like(T, spt))
            for _ in range(2):
                o = torch.fmod(torch.full_like(T, D), T)
                N = ((D - o) / T).round()
                need = torch.where(N > 0, o + T, o).floor() + 2
                T = torch.where(need > cap, torch.full_like(T, spt), T)
            return T, o, N, need

        rows = [(R, V)]
        if T is not None:
            T, o, N, need = decompose(T)
            for _ in range(int(need.max().item())):
                rows.append(self.fine(*rows[-1], self.h))
            return rows, T, o, N
        ne = torch.zeros_like(R)
        t1, T = torch.zeros_like(R), torch.full_like(R, spt)
        need = torch.full_like(R, float("inf"))
        o = N = None
        for k in range(1, cap + 1):
            rows.append(self.fine(*rows[-1], self.h))
            if k >= 2:
                v0, v1, v2 = rows[k - 2][1], rows[k - 1][1], rows[k][1]
                hit = ((v0 > 0) != (v1 > 0)) & (ne < 3)
                t = (k - 2) + self.root(v0, v1, v2)
                ne = ne + hit
                t1 = torch.where(hit & (ne == 1), t, t1)
                third = hit & (ne == 3)
                T = torch.where(third, t - t1, T)
                need = torch.where(third, torch.zeros_like(R) if detect else decompose(T)[3], need)
                if k >= 100 and bool((need <= k).all()):
                    break
        if not detect:
            T, o, N, need = decompose(T)
            while len(rows) <= int(need.max().item()):
                rows.append(self.fine(*rows[-1], self.h))
        return rows, T, o, N

    def periods(self, R, V):
        return self.window(R, V, detect=True)[1]

    def etd(self, R, V, T=None):
        rows, T, o, N = self.window(R, V, T)
        Rs, Vs = torch.stack([r for r, _ in rows]), torch.stack([v for _, v in rows])

        def land(u):
            k = u.floor()
            s, k = u - k, k.long()
            return tuple((lambda a, b, c: a + s * ((-3 * a + 4 * b - c) / 2 + s * ((a - 2 * b + c) / 2)))(
                *(Y.gather(0, (k + q).clamp(max=len(rows) - 1)[None])[0] for q in range(3))) for Y in (Rs, Vs))

        y0, y1 = land(o), land(torch.where(N > 0, o + T, o))
        return tuple(a + N * (b - a) for a, b in zip(y0, y1)), T, o, N

    def classic(self, R, V, modified):
        P = 2 * math.pi * self.eps if not modified else self.periods(R, V).mean().item() * self.h
        o = math.fmod(self.c["dt"], P)
        N = round((self.c["dt"] - o) / P)
        if modified:
            r, v = self.advance(R, V, P)
        else:
            r, v = R, V
            for _ in range(self.spt):
                r, v = self.fine(r, v, self.h)
        return (*self.advance(R + N * (r - R), V + N * (v - V), o), P)


def _bf16(x):
    return x.float().bfloat16().double()


def _gelu(u):
    return 0.5 * u * torch.erfc(-u / math.sqrt(2))


def _gelu_d(u):
    return 0.5 * torch.erfc(-u / math.sqrt(2)) + u * torch.exp(-0.5 * u * u) / math.sqrt(2 * math.pi)


def _weights(w):
    out, k = [], 0
    for _, shape in inputs.MLP_SHAPES:
        m = int(np.prod(shape))
        out.append(w[k : k + m].reshape(shape))
        k += m
    return out


def _net(w, X):
    """The network with its bfloat16 rounding points."""
    W1, b1, W2, b2, W3, b3 = _weights(w)
    z1 = X @ _bf16(W1).T + b1
    h1 = _bf16(_gelu(z1))
    z2 = h1 @ _bf16(W2).T + b2
    h2 = _bf16(_gelu(z2))
    return h2 @ _bf16(W3).T + b3, z1, h1, z2, h2


def _net_grad(w, X, T):
    _, _, W2, _, W3, _ = _weights(w)
    out, z1, h1, z2, h2 = _net(w, X)
    d = out - T
    dout = d / X.shape[0]
    dz2 = (dout @ _bf16(W3)) * _gelu_d(z2)
    dz1 = (_bf16(dz2) @ _bf16(W2)) * _gelu_d(z1)
    grads = [dz1.T @ X, dz1.sum(0), _bf16(dz2).T @ h1, dz2.sum(0), dout.T @ h2, dout.sum(0)]
    return torch.cat([g.reshape(-1) for g in grads]), (d * d).sum().item() / (2 * X.shape[0])


def _exact_learned(c, R, V, seed):
    b = _Beam(c)
    E, edges = b.node_field(b.charge(R), R.numel())
    k = b.nc // 2
    psi = torch.cat([torch.zeros(1, dtype=torch.float64, device="cuda"), (0.5 * b.hr * (E[1:] + E[:-1])).cumsum(0)])
    psi = psi - psi[k]

    def H(r, v):
        inside, j, f, below = b.locate(r)
        d = f * b.hr
        p = psi[j] + E[j] * d + (E[j + 1] - E[j]) * d * d / (2 * b.hr)
        out = torch.where(below, psi[0] + edges[0] * torch.log(r / b.rm), psi[-1] + edges[1] * torch.log(r / -b.rm))
        return 0.5 * (r * r + v * v) - c["eps"] * torch.where(inside, p, out)

    (r, v), _, _, _ = b.etd(R, V)
    one = torch.ones_like(R)
    w = torch.from_numpy(inputs.mlp_init(seed)).double().cuda()
    out = _net(w, torch.stack([R, V, 0 * one, one, c["dt"] * one], dim=1).float().double())[0]
    rl, vl = r + _scale()[0] * out[:, 0], v + _scale()[1] * out[:, 1]
    h0 = H(r, v)
    keep = (H(rl, vl) - h0).abs() <= c["tol"] * h0.abs()
    return {"r": torch.where(keep, rl, r), "v": torch.where(keep, vl, v), "more": None}


def _exact_step(c, R, V):
    b = _Beam(c)
    more = None
    T = b.periods(R, V) if c["once"] else None
    for _ in range(c["steps"] if c["scheme"] != "fine" else 1):
        if c["scheme"] == "etd":
            R, V = b.etd(R, V, T)[0]
        elif c["scheme"] == "fine":
            R, V = b.advance(R, V, 2 * math.pi * c["eps"] * 1.005)
        else:
            R, V, more = b.classic(R, V, c["scheme"] == "modified")
    return {"r": R, "v": V, "more": more}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("step", "learned", "diag"):
        if c["n"] * c["steps"] > 3_000_000:  # minutes of plain FP64
            return None
        R, V = _beam(c["beam"], c["n"], seed, c["precision"])
        if kind == "step":
            return _exact_step(c, R, V)
        if kind == "learned":
            return _exact_learned(c, R, V, seed)
        b = _Beam(c)
        (R, V), T, o, N = b.etd(R, V)
        n = R.numel()
        E, edges = b.node_field(b.charge(R), n)
        m = {"charge": 1.0, "kinetic": 0.5 * (R * R + V * V).mean(), "mean_R": R.mean(), "mean_V": V.mean(), "rms_R": (R * R).mean().sqrt(),
             "rms_V": (V * V).mean().sqrt(), "T_min": T.min() * b.h, "T_mean": T.mean() * b.h, "T_max": T.max() * b.h}
        return {"m": {k: float(x) for k, x in m.items()}, "Q": None, "E": E, "edges": edges, "n_out": None, "T": T * b.h, "N": None, "o": o * b.h}
    if kind == "batch":
        beams = _batch_cases(c, seed)
        got = [_exact_step(b, *_beam(b["beam"], b["n"], seed + i, 1)) for i, b in enumerate(beams)]
        return [(g["r"], g["v"]) for g in got]
    if kind == "mesh":
        b = _Beam(dict(STEP, **dict(GAUSS, n_cells=c["n_cells"], r_max=c["r_max"])))
        R = _beam("wide", c["n"], seed, c["precision"])[0]
        E, edges = b.node_field(b.charge(R), c["n"])
        return {"Q": None, "n_out": None, "E": E, "edges": edges, "e": b.at(E, edges, R)}
    if kind == "forward":
        X, _ = _samples(c["n"], seed)
        return _net(torch.from_numpy(inputs.mlp_init(seed)).double().cuda(), X.double())[0]
    X, T = _samples(c["n"], seed)
    n, batch = c["n"], min(c["batch"], c["n"])
    mul = max(1, int(n * 0.6180339887498949))  # the library's walk through the data set, seed 0
    while math.gcd(mul, n) != 1:
        mul += 1
    w = torch.from_numpy(inputs.mlp_init(seed)).double().cuda()
    m, v, hist = torch.zeros_like(w), torch.zeros_like(w), []
    for t in range(1, c["steps"] + 1):
        at = (((t - 1) * batch % n + torch.arange(batch, device="cuda")) % n * mul) % n
        g, loss = _net_grad(w, X[at].double(), T[at].double())
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        w = w - 1e-3 * (m / (1 - 0.9**t)) / ((v / (1 - 0.999**t)).sqrt() + 1e-8)
        hist.append(loss)
    g, loss = _net_grad(w, X[:batch].double(), T[:batch].double())
    return {"w": w, "hist": torch.tensor(hist), "grad": g, "loss": loss}
