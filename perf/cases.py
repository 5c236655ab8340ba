"""The performance cases of the framework: what a user has it compute, through
its public entry points (``native.Gap``, ``Batch``, ``Gap2D``, the ``cp_mlp_*``
training calls and the allocation-free ion push).

Kinds of case
  step      one time step and the level's scalars, of a gap that has been
            running for a while: a host loop that looks at every level.
  run       a whole job: create the gap, load its plasma, advance it from
            t = 0, read every level's diagnostics and the final grid.
  steady    a stretch of levels of a long run past the beam's transit (ion
            impacts and secondary emission every step), and its read-out.
  ensemble  the same for many uneven independent gaps advanced together.
  gap2d     a stretch of levels of the 2D planar gap and its fields.
  train     one step of the predictor's training: loss, gradient, Adam.
  ions      the allocation-free push of one ion population.

Read-outs leave out ``residual`` (the solve's backward error: rounding noise)
and the particle stores (their order is unspecified; the integer charge grid
holds every particle's position to 2^-16 of a cell).
"""
import math

import numpy as np
import torch

from paper_2603_24010_gb300 import native
from paper_2603_24010_gb300 import workloads as W

MODES = {"strict": native.STRICT, "weak": native.WEAK, "learned": native.WEAK_LEARNED}
FLOATS = ("V_gap", "I_circ", "Q_surf", "Q_conv", "Q_circ", "V_source", "ion_energy_eV", "max_cfl", "J_hat")
WHOLE = ("absorbed", "emitted", "injected", "n_live", "conv_count")


def listed():
    return [
        # the smallest call: one strict step of the FP64 gap, its scalars read back
        dict(name="step_fp64", kind="step", cells=256, pairs=10_000, beam=50, beam_mode=0, dt_ps=1.0,
             precision="fp64", mode="strict", advance=3000),
        # the small FP64 gap as a whole job (FP64 particles, uniform beam spectrum)
        dict(name="run_fp64", kind="run", workload="gap", cells=256, pairs=10_000, beam=50, beam_mode=1,
             dt_ps=1.0, precision="fp64", mode="strict", steps=1000),
        # the paper's integrated configuration: Tesla transformer, heavy ions, sampled SEE laws
        dict(name="run_tesla", kind="run", workload="tesla", cells=600, pairs=500, beam=20, beam_mode=0,
             dt_ps=15000.0, precision="fp64", mode="weak", steps=575),
        # a middle-sized FP32 job of ragged size, plain weak coupling
        dict(name="run_ragged", kind="run", workload="gap", cells=1531, pairs=333_337, beam=331, beam_mode=1,
             dt_ps=0.75, precision="fp32", mode="weak", steps=701),
        # the large FP32 gap from t = 0 (1e7 macroparticles, about the L2's size)
        dict(name="run_large", kind="run", workload="gap", cells=4096, pairs=5_000_000, beam=5000, beam_mode=0,
             dt_ps=0.5, precision="fp32", mode="strict", steps=640),
        # the large FP32 gap at steady state: about 3e7 macroparticles, impacts every step
        dict(name="steady_large", kind="steady", cells=4096, pairs=5_000_000, beam=5000, beam_mode=0, dt_ps=0.5,
             precision="fp32", mode="strict", advance=12_000, steps=128),
        # the 100 x thinned large gap with the learned predictor in the loop
        dict(name="steady_learned", kind="steady", cells=4096, pairs=50_000, beam=50, beam_mode=0, dt_ps=0.5,
             precision="fp32", mode="learned", advance=6000, steps=256),
        # a parameter scan: uneven gaps advanced as one ensemble
        dict(name="ensemble", kind="ensemble", instances=160, thin=2, max_cells=4096, mode="strict",
             advance=2560, steps=256),
        # the 2D gap at a test's size, and at the benchmark's grid with a fifth of its particles
        dict(name="gap2d_small", kind="gap2d", nx=96, ny=128, pairs=150_000, beam=150, mode="weak", steps=64),
        dict(name="gap2d_large", kind="gap2d", nx=1024, ny=1024, pairs=10_000_000, beam=2000, mode="strict",
             steps=96),
        # the predictor's training step at its default mini-batch
        dict(name="train_step", kind="train", batch=8192),
        # the allocation-free push at the largest population it takes
        dict(name="ions_noalloc", kind="ions", cells=4096, ions=524_288),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("step", "run", "run", "run", "steady", "steady", "ensemble", "gap2d", "gap2d", "train",
                       "ions"))
    mode = rng.choice(("strict", "weak"))
    if kind == "train":
        return dict(kind=kind, batch=_log(rng, 257, 65_536))
    if kind == "ions":
        return dict(kind=kind, cells=_log(rng, 16, 4096), ions=_log(rng, 1000, 524_288))
    if kind == "ensemble":
        return dict(kind=kind, instances=_log(rng, 2, 160), thin=rng.choice((2, 3, 10)),
                    max_cells=_log(rng, 300, 4096), mode=mode, advance=_log(rng, 200, 2560),
                    steps=rng.choice((64, 100, 256)))
    if kind == "gap2d":
        pairs = _log(rng, 20_000, 4_000_000)
        return dict(kind=kind, nx=_log(rng, 40, 1024), ny=rng.choice((8, 64, 128, 256, 512, 1024)), pairs=pairs,
                    beam=rng.choice((0, pairs // 5000, pairs // 2000)), mode=mode, steps=rng.choice((16, 33, 64)))
    precision = rng.choice(("fp64", "fp32", "fp32", "fp32"))
    pairs = _log(rng, 500, 500_000 if precision == "fp64" else 3_000_000)
    case = dict(kind=kind, cells=_log(rng, 64, 4096), pairs=pairs, beam=rng.choice((0, 1 + pairs // 1000)),
                beam_mode=rng.choice((0, 1)), dt_ps=rng.choice((0.5, 1.0)), precision=precision, mode=mode)
    if kind == "run":
        return dict(case, workload="gap", steps=_log(rng, 100, 700))
    case["advance"] = _log(rng, 100, 3000)
    if kind == "steady":
        case.update(steps=rng.choice((64, 100, 256)), mode=rng.choice(("strict", "weak", "learned")))
    return case


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _cfg(case, seed):
    """The workload dictionary of a single 1D gap."""
    if case.get("workload") == "tesla":
        cfg = W.scaled(W.tesla_gap(seed), n_cells=case["cells"], n_pairs=case["pairs"],
                       beam_per_step=case["beam"])
        cfg["weight"] = W.tesla_gap()["weight"] * 500 / case["pairs"]
    else:
        cfg = W.scaled(W.gap_1d_fp32_large(seed), n_cells=case["cells"], n_pairs=case["pairs"],
                       beam_per_step=case["beam"], beam_mode=case["beam_mode"], dt=case["dt_ps"] * 1e-12)
        cfg["weight"] = cfg["n0"] * cfg["d"] * cfg["area"] / cfg["n_pairs"]
    cfg["precision"] = W.FP64 if case["precision"] == "fp64" else W.FP32
    return cfg


def _persistence_net(cfg):
    """A network that predicts the next level's plasma charge to be the last one's (what a trained one
    does to first order): identity chains through the three hidden layers, whose GELU is linear at 40."""
    S = 10.0 * cfg["e"] * cfg["weight"]
    p = np.zeros(native.MLP_NPARAM, np.float32)
    w1 = p[:2560].reshape(64, 40)
    w1[0, 35:38] = (1.0, 1.0, -1.0)
    p[2560] = 40.0
    p[2624] = p[6784] = 1.0  # W2[0, 0], W3[0, 0]
    p[10944 + 64] = 1.0      # W4[1, 0]
    p[11073] = -40.0
    norm = native.cp_predictor(bound=0.5)
    norm.in_scale[:] = (S, S / cfg["C"], S, 1.0, 1.0)
    norm.out_scale[:] = (1.0, S)
    return p, norm


def _stores(pairs, beam, dt_ps):
    """Store capacities of a gap that runs on and on: the plasma and the beam ions in flight (the slowest,
    of 5 keV, cross in 5.1 ns), and as many secondaries."""
    n = int(1.2 * (pairs + beam * (6000 / dt_ps + 256))) + 65_536
    return (0, n, n)


def _running_gap(case, seed, max_steps):
    cfg = _cfg(case, seed)
    g = native.Gap(cfg, capacity=_stores(case["pairs"], case["beam"], case["dt_ps"]), max_steps=max_steps)
    g.load_species(case["pairs"], cfg["T_load_eV"], seed)
    if case["mode"] == "learned":
        g.set_predictor(*_persistence_net(cfg))
    g.step(MODES[case["mode"]], case["advance"])
    return g


def _cfg2d(case, seed):
    cfg = W.gap_2d(seed, Nx=case["nx"], Ny=case["ny"], n_pairs=case["pairs"], beam_per_step=case["beam"])
    return cfg


def _train_inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def normal(*shape):
        return torch.randn(shape, device="cuda", generator=gen)

    n, P = case["batch"], native.MLP_NPARAM
    # windows of 8 levels of 5 features: a slow part and a level's own noise, unit scale
    X = (0.8 * normal(n, 1, 5) + 0.6 * normal(n, 8, 5)).reshape(n, 40).contiguous()
    Y = 0.5 * X[:, 35:37] + 0.5 * normal(n, 2)
    m = 1e-3 * normal(P)
    v = 1e-5 * (0.5 + torch.rand(P, device="cuda", generator=gen))
    return X, Y.contiguous(), m, v


TRAIN_T, TRAIN_LR = 100, 1e-3


def _ion_inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    N, n = case["cells"], case["ions"]
    cfg = W.scaled(W.gap_1d_fp32_large(seed), n_cells=N, dt=1e-12, see_scale=8.0)
    x = (torch.rand(n, device="cuda", generator=gen) * N).clamp(1e-3, N - 0.01 * N / 4096 - 1e-3)
    u = torch.randn(n, device="cuda", generator=gen) * W.thermal_u(cfg, cfg["m_i"], 50.0)
    ids = torch.randperm(n, device="cuda", generator=gen).to(torch.int32)
    E = 1e4 * torch.randn(N, device="cuda", generator=gen, dtype=torch.float64)
    return cfg, x, u, ids, E


def prepare(case, seed):
    kind = case["kind"]
    if kind == "run":
        return dict(case=case, cfg=_cfg(case, seed), seed=seed)
    if kind == "step":
        return dict(case=case, gap=_running_gap(case, seed, case["advance"] + 150_000))
    if kind == "steady":
        return dict(case=case, gap=_running_gap(case, seed, case["advance"] + 3000 * case["steps"]))
    if kind == "ensemble":
        cfgs = [W.scaled(c, seed=(seed * 1009 + i) & 0x7FFFFFFF) for i, c in enumerate(
            W.ensemble(case["instances"], 0, thin=case["thin"], n_cells_max=case["max_cells"]))]
        b = native.Batch(cfgs, max_steps=case["advance"] + (300 if len(cfgs) > 64 else 1500) * case["steps"],
                         capacity=_stores(max(c["n_pairs"] for c in cfgs),
                                          max(c["beam_per_step"] for c in cfgs), 1.0))
        for i, c in enumerate(cfgs):
            xi, ue, ui = W.load_pairs(c)
            b.set_particles(i, native.ELECTRONS, xi, ue)
            b.set_particles(i, native.IONS, xi, ui)
        _ok(b.step(MODES[case["mode"]], case["advance"]))
        return dict(case=case, batch=b)
    if kind == "gap2d":
        cfg = _cfg2d(case, seed)
        xi, eta, ue, we, ui, wi = W.load_pairs_2d(cfg)
        g = native.Gap2D(cfg, max_steps=3000 * case["steps"], capacity=_stores(case["pairs"], case["beam"], 1.0))
        g.set_particles(native.ELECTRONS, xi, eta, ue, we)
        g.set_particles(native.IONS, xi, eta, ui, wi)
        g.step(MODES[case["mode"]], 0)  # the stores, and level 0
        return dict(case=case, gap=g)
    if kind == "train":
        X, Y, m, v = _train_inputs(case, seed)
        f = dict(dtype=torch.float32, device="cuda")
        s = dict(case=case, X=X, Y=Y, m=m, v=v, t=TRAIN_T, params=torch.empty(native.MLP_NPARAM, **f),
                 grad=torch.empty(native.MLP_NPARAM, **f), loss=torch.empty(1, **f),
                 work=torch.empty(native.cp_mlp_work_floats(), **f))
        _ok(native.cp_mlp_init(s["params"].data_ptr(), seed, native.current_stream()))
        return s
    cfg, x, u, ids, E = _ion_inputs(case, seed)
    gap, _, see, _ = native.structs_from_config(cfg)
    cap = 4 * case["ions"] + 64
    return dict(case=case, cfg=cfg, gap=gap, see=see, xi=x, u=u, ids=ids, E=E, cap=cap,
                G=torch.empty(case["cells"] + 1, dtype=torch.int64, device="cuda"),
                se_xi=torch.empty(cap, device="cuda"), se_u=torch.empty(cap, device="cuda"),
                counts=torch.empty(6, dtype=torch.int64, device="cuda"))


def _ok(rc):
    if rc != native.OK:
        raise native.CpError("case", rc)


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _columns(h):
    return {k: h[k] for k in FLOATS + WHOLE}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        g = state["gap"]
        g.step(MODES[case["mode"]], 1)
        d = g.scalars()
        return dict({k: getattr(d, k) for k in FLOATS}, n_live=list(d.n_live), conv_count=d.conv_count,
                    injected=d.injected, emitted=list(d.emitted))
    if kind == "run":
        cfg = state["cfg"]
        g = native.Gap(cfg, max_steps=case["steps"])
        g.load_species(case["pairs"], cfg["T_load_eV"], state["seed"])
        g.step(MODES[case["mode"]], case["steps"])
        out = dict(history=_columns(g.history()), grid=g.grid())
        g.close()
        return out
    if kind == "steady":
        g = state["gap"]
        g.step(MODES[case["mode"]], case["steps"])
        return dict(history=_columns(g.history(g.level + 1 - case["steps"], case["steps"])), grid=g.grid())
    if kind == "ensemble":
        b, n = state["batch"], case["steps"]
        _ok(b.step(MODES[case["mode"]], n))
        first = b.level + 1 - n
        hs = [_columns(b.history(i, first, n)) for i in range(b.n)]
        gs = [b.grid(i) for i in range(b.n)]
        return dict(history={k: np.stack([h[k] for h in hs]) for k in hs[0]},
                    grid={k: np.concatenate([g[k] for g in gs]) for k in gs[0]})
    if kind == "gap2d":
        g = state["gap"]
        g.step(MODES[case["mode"]], case["steps"])
        return dict(history=_columns(g.history(g.level + 1 - case["steps"], case["steps"])), fields=g.fields())
    st = native.current_stream()
    if kind == "train":
        p = {k: state[k].data_ptr() for k in ("params", "X", "Y", "grad", "loss", "work", "m", "v")}
        _ok(native.cp_mlp_loss_grad(p["params"], p["X"], p["Y"], case["batch"], p["grad"], p["loss"], p["work"],
                                    st))
        _ok(native.cp_mlp_adam(p["params"], p["grad"], p["m"], p["v"], state["t"], TRAIN_LR, stream=st))
        state["t"] += 1
        return {k: state[k] for k in ("params", "grad", "loss", "m", "v")}
    # emitted electrons come in no fixed order; their number and (in G) their charge come back
    _ok(native.cp_push_ions_noalloc(state["gap"], state["see"], state["cfg"]["dt"], state["cfg"]["seed"], 7, 0,
                                    state["E"].data_ptr(), state["xi"].data_ptr(), state["u"].data_ptr(),
                                    state["ids"].data_ptr(), case["ions"], state["G"].data_ptr(),
                                    state["se_xi"].data_ptr(), state["se_u"].data_ptr(), state["cap"],
                                    state["counts"].data_ptr(), st))
    return {k: state[k] for k in ("xi", "u", "G", "counts")}


# ---------------------------------------------------------------------------
# The work of one pass: particles read and written once a step, grids and
# diagnostics written once; the kick, drift, gather and deposit of each
# ---------------------------------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "train":
        n = case["batch"]
        macs = 40 * 64 + 2 * 64 * 64 + 64 * 2
        return dict(bytes=4.0 * (42 * n + 7 * native.MLP_NPARAM), flops=6.0 * macs * n)
    if kind == "ions":
        return dict(bytes=20.0 * case["ions"] + 16.0 * case["cells"], flops=20.0 * case["ions"])
    steps = case.get("steps", 1)
    if kind == "gap2d":
        live = 2 * case["pairs"] + case["beam"] * steps / 2
        nodes = (case["nx"] + 1) * case["ny"]
        return dict(bytes=steps * (32.0 * live + 24.0 * nodes),
                    flops=steps * (60.0 * live + 20.0 * nodes * math.log2(case["ny"])))
    if kind == "ensemble":
        cfgs = W.ensemble(case["instances"], 0, thin=case["thin"], n_cells_max=case["max_cells"])
        live = sum(c["n_pairs"] * 2 + c["beam_per_step"] * min(case["advance"], 2500) for c in cfgs)
        return dict(bytes=steps * 16.0 * live, flops=steps * 20.0 * live)
    b = 32.0 if case["precision"] == "fp64" else 16.0
    transit = 2550.0 / case["dt_ps"]  # steps a 20 keV ion takes across the gap
    levels = min(case.get("advance", steps / 2), transit)
    live = 2 * case["pairs"] + case["beam"] * levels
    return dict(bytes=steps * (b * live + 200.0 + 24.0 * case["cells"]), flops=steps * 20.0 * live)


# ---------------------------------------------------------------------------
# Reference values in 64 bits: the definitions in plain torch
# ---------------------------------------------------------------------------
_M32 = 0xFFFFFFFF


def _s64(v):
    v &= (1 << 64) - 1
    return v - (1 << 64) if v >> 63 else v


def _philox(c0, c1, c2, seed, tag):
    """Philox4x64-10 words of counters (c0, c1, c2, 0) under key (seed, tag); int64 tensors hold the bits."""
    def mul(a, m):
        al, ah, ml, mh = a & _M32, (a >> 32) & _M32, m & _M32, m >> 32
        p0, p1, p2 = al * ml, ah * ml, al * mh
        t = ((p0 >> 32) & _M32) + (p1 & _M32) + (p2 & _M32)
        hi = ah * mh + ((p1 >> 32) & _M32) + ((p2 >> 32) & _M32) + ((t >> 32) & _M32)
        return hi, a * _s64(m)

    c3, k0, k1 = torch.zeros_like(c0), seed, tag
    for _ in range(10):
        h0, l0 = mul(c0, 0xD2E7470EE14C6C93)
        h1, l1 = mul(c2, 0xCA5A826395121157)
        c0, c1, c2, c3 = h1 ^ c1 ^ _s64(k0), l1, h0 ^ c3 ^ _s64(k1), l0
        k0, k1 = k0 + 0x9E3779B97F4A7C15, k1 + 0xBB67AE8584CAA73B
    return c0, c1, c2, c3


def _u01(w):
    return (((w >> 12) & ((1 << 52) - 1)).double() + 0.5) * 2.0 ** -52


def _normal(ua, ub):
    return torch.sqrt(-2 * torch.log(ua)) * torch.cos(2 * math.pi * ub)


class _Sim:
    """The circuit-coupled gap in 64 bits, one (y periodic: two) dimension(s), from its definition."""

    def __init__(self, cfg, mode, dev, ny=0):
        self.c, self.mode, self.dev, self.ny = cfg, mode, dev, ny
        self.N, self.dt, self.A = int(cfg["n_cells"]), cfg["dt"], cfg["area"]
        self.dx = cfg["d"] / self.N
        self.dy = cfg["Ly"] / ny if ny else 0.0
        self.fix = 2.0 ** (32 if ny else 16)
        self.alpha = self.dx * cfg["e"] * cfg["weight"] / (self.A * self.fix * cfg["eps0"])
        self.mass = (cfg["m_e"], cfg["m_i"], cfg["m_e"])
        self.charge = (-1, 1, -1)
        z = torch.zeros(0, dtype=torch.float64, device=dev)
        self.p = [[z, z, z, z] for _ in range(3)]  # x, u, y, w
        self.ids = torch.zeros(0, dtype=torch.int64, device=dev)
        self.Q, self.sigma, self.phi0, self.level, self.pushed = [0.0] * 4, cfg["sigma0"], 0.0, 0, False
        self.tesla = cfg.get("circuit") == 2
        if self.tesla:
            self.Qt = [np.array([cfg["tC1"] * cfg["tV1"], 0, 0, 0, 0.0])] * 4
        self.rows = {k: [] for k in FLOATS}

    # -- circuit: Q^n = K - g phi_0^n ----------------------------------------
    def _loops(self, first):
        """The Tesla loops' next charges as K - phi_0 g (all five)."""
        c, dt = self.c, self.dt
        a, b = 1.5 / dt, 2.25 / dt ** 2
        if first:
            return self.Qt[0], np.zeros(5)
        R1, R2, R3, M = c["tR1"], c["tR2"], c["tR3"], c["tM"]
        strict = self.mode == "strict"
        T = np.array([[1 / c["tC1"] + a * R1, -a * R1, 0, 0, -a * R1],
                      [-a * R1, a * (R1 + R2) + b * c["tL1"], b * M, 0, a * R1],
                      [0, b * M, b * c["tL2"] + a * R3, -a * R3, a * R3],
                      [0, 0, -a * R3, a * R3 + (0 if strict else 1 / c["tC3"]), -a * R3],
                      [-a * R1, a * R1, a * R3, -a * R3, a * (R1 + R3) + 1 / c["tC2"]]])
        q = self.Qt
        d1, d2 = (4 * q[0] - q[1]) / (2 * dt), (24 * q[0] - 22 * q[1] + 8 * q[2] - q[3]) / (4 * dt ** 2)
        x1, x3 = d1[0] - d1[1] - d1[4], d1[2] - d1[3] + d1[4]
        r = np.array([R1 * x1, -R1 * x1 + R2 * d1[1] + c["tL1"] * d2[1] + M * d2[2],
                      M * d2[1] + c["tL2"] * d2[2] + R3 * x3, -R3 * x3, -R1 * x1 + R3 * x3])
        if not strict:
            r[3] += self.Q[0] / c["tC3"] - self.phi0
        K = np.linalg.solve(T, r)
        return K, np.linalg.solve(T, np.eye(5)[3]) if strict else np.zeros(5)

    def _circuit(self, first):
        c, dt, Q = self.c, self.dt, self.Q
        if self.tesla:
            K, g = self._loops(first)
            self._K5, self._g5 = K, g
            return K[3], g[3], 0.0
        t = self.level * dt
        Vs = c["polarity"] * c["V0"] * (1 - math.cos(2 * math.pi * c["f"] * t)) * math.exp(-t / c["tau"]) / 2
        a21 = 2.25 * c["L"] / dt ** 2 + 1.5 * c["R"] / dt
        hist = (c["L"] * (24 * Q[0] - 22 * Q[1] + 8 * Q[2] - Q[3]) / (4 * dt ** 2)
                + c["R"] * (4 * Q[0] - Q[1]) / (2 * dt))
        if self.mode == "strict":
            return (Vs + hist) / a21, 1 / a21, Vs
        return (Vs + hist + Q[0] / c["C"] - self.phi0) / (a21 + 1 / c["C"]), 0.0, Vs

    # -- deposit and solve ------------------------------------------------------
    def _deposit(self):
        N, ny = self.N, max(self.ny, 1)
        G = torch.zeros((N + 1) * ny, dtype=torch.int64, device=self.dev)
        for s in range(3):
            x, _, y, _ = self.p[s]
            i = torch.floor(x).long()
            wx = torch.floor((x - i) * 65536.0).long()
            cells = [(i, 65536 - wx), (i + 1, wx)]
            if self.ny:
                j = torch.floor(y).long()
                wy = torch.floor((y - j) * 65536.0).long()
                cells = [(a * ny + b % ny, wa * wb) for a, wa in cells for b, wb in ((j, 65536 - wy), (j + 1, wy))]
            for k, w in cells:
                G.index_add_(0, k, self.charge[s] * w)
        G = G.reshape(N + 1, ny)
        G[0] *= 2
        G[N] *= 2
        return G

    def _solve(self, first, conv, energy, cfl):
        c, N = self.c, self.N
        G = self._deposit()
        G1 = G.sum(1)
        K, g, Vs = self._circuit(first)
        Qconv = conv * c["e"] * c["weight"]
        gam = g * self.dx / (c["eps0"] * self.A)
        b0 = self.dx / c["eps0"] * (self.sigma + (Qconv + K - self.Q[0]) / self.A) + self.alpha * float(G1[0]) / 2
        S = G1[:N].clone()
        S[0] = 0
        S = torch.cumsum(S, 0)
        phi0 = (N * b0 + self.alpha * float(S.double().sum())) / (1 + N * gam)
        D = (b0 - gam * phi0) + self.alpha * S.double()
        phi = torch.zeros(N + 1, dtype=torch.float64, device=self.dev)
        phi[:N] = torch.flip(torch.cumsum(torch.flip(D, [0]), 0), [0])
        Qn = K - g * phi0
        if self.tesla and not first:
            self.Qt = [self._K5 - phi0 * self._g5] + self.Qt[:3]
        I = (3 * Qn - 4 * self.Q[0] + self.Q[1]) / (2 * self.dt)
        self.sigma += (Qconv + Qn - self.Q[0]) / self.A
        self.Q = [Qn] + self.Q[:3]
        self.phi0 = phi0
        for k, v in zip(FLOATS, (phi0, I, self.sigma * self.A, Qconv, Qn, Vs, energy, cfl, 0.0)):
            self.rows[k].append(v)
        self.G, self.phi, self.E = G, phi, D / self.dx
        if self.ny:
            self._transverse(G)

    def _transverse(self, G):
        """k != 0 modes: sine transform in x, Fourier in y of the five-point equation, zero on both electrodes."""
        c, N, ny = self.c, self.N, self.ny
        rho = (G.double() - G.double().mean(1, keepdim=True))[1:N] * (
            c["e"] * c["weight"] / (self.dx * self.dy * (self.A / c["Ly"]) * self.fix))
        i = torch.arange(1, N, dtype=torch.float64, device=self.dev)
        S = math.sqrt(2.0 / N) * torch.sin(math.pi / N * torch.outer(i, i))
        lx = 2 - 2 * torch.cos(math.pi / N * i)
        k = torch.arange(ny // 2 + 1, dtype=torch.float64, device=self.dev)
        ly = (self.dx / self.dy) ** 2 * (2 - 2 * torch.cos(2 * math.pi / ny * k))
        F = torch.fft.rfft(S @ rho, dim=1) * (self.dx ** 2 / c["eps0"]) / (lx[:, None] + ly[None, :])
        F[:, 0] = 0
        pt = torch.zeros(N + 1, ny, dtype=torch.float64, device=self.dev)
        pt[1:N] = S @ torch.fft.irfft(F, n=ny, dim=1)
        self.Ex = self.E[:, None] + (pt[:-1] - pt[1:]) / self.dx
        self.Ey = (pt - torch.roll(pt, -1, 1)) / self.dy
        self.phi2 = self.phi[:, None] + pt

    # -- particles ------------------------------------------------------------
    def _gather(self, x, y):
        N, ny = self.N, self.ny
        s = x - 0.5
        i = torch.floor(s).clamp(0, N - 1)
        t = (s - i).clamp(0, 1)
        i = i.long()
        t = torch.where(i >= N - 1, torch.zeros_like(t), t)
        i1 = (i + 1).clamp(max=N - 1)
        if not ny:
            return self.E[i] + t * (self.E[i1] - self.E[i]), None

        def bilin(F, i, i1, t, y):
            j = torch.floor(y)
            v = y - j
            j, j1 = j.long() % ny, (j.long() + 1) % ny
            return (1 - v) * ((1 - t) * F[i, j] + t * F[i1, j]) + v * ((1 - t) * F[i, j1] + t * F[i1, j1])

        a = torch.floor(x)
        return bilin(self.Ex, i, i1, t, y), bilin(self.Ey, a.long(), a.long() + 1, x - a, y - 0.5)

    def _emit(self, hits):
        """Secondary electrons of the absorbed ions: (ids, electrode, u, w, y)."""
        c, dt = self.c, self.dt
        ids, el, u, w, y = hits
        E = 0.5 * c["m_i"] * ((u * self.dx / dt) ** 2 + (w * self.dy / dt) ** 2) / c["e"]
        gam = (c["see_scale"] * c["gamma_coef"] * torch.sqrt(E / c["E_ref_eV"])).clamp(max=c["gamma_max"])
        step = torch.full_like(ids, self.level)
        u1 = _u01(_philox(ids, step, torch.zeros_like(ids), c["seed"], 0x5345)[0])
        if c["see_count_law"] == 1:
            n = torch.zeros_like(ids)
            pk = torch.exp(-gam)
            F = pk.clone()
            for k in range(1, 65):
                n += (u1 >= F).long()
                pk = pk * gam / k
                F += pk
        else:
            n = (torch.floor(gam) + (u1 < gam - torch.floor(gam)).double()).long()
        energy = float(torch.round(E * 256)[el == 0].sum()) / 256
        conv = int(n[el == 0].sum())
        r = torch.repeat_interleave(torch.arange(ids.numel(), device=self.dev), n)
        j = torch.arange(r.numel(), device=self.dev) - (torch.cumsum(n, 0) - n)[r]
        wv = _philox(ids[r], step[r], 1 + j, c["seed"], 0x5345)
        z = _normal(_u01(wv[0]), _u01(wv[1]))
        if c["see_energy_law"] == 1:
            v = torch.sqrt(2 * torch.exp(c["see_ln_mu"] + c["see_ln_sigma"] * z) * c["e"] / c["m_e"])
        else:
            v = math.sqrt(c["e"] * c["T_emit_eV"] / c["m_e"]) * z.abs()
        us = v * dt / self.dx
        low = el[r] == 0
        x = torch.where(low, us * _u01(wv[2]), self.N - us * _u01(wv[2]))
        self._append(2, x, torch.where(low, us, -us), y[r], torch.zeros_like(us))
        return conv, energy

    def _append(self, s, x, u, y, w):
        x = x.clamp(1e-300, math.nextafter(self.N, 0))
        self.p[s] = [torch.cat(q) for q in zip(self.p[s], (x, u, y, w))]

    def _beam(self, steps):
        """The beam's draws of `steps` levels: position, speed and transverse position, a row a level."""
        c, B = self.c, int(self.c["beam_per_step"])
        k = torch.arange(B, device=self.dev).repeat(steps)
        n = torch.arange(steps, device=self.dev).repeat_interleave(B) + self.level
        wv = _philox(k, n, torch.zeros_like(k), c["seed"], 0x4245)
        Eb = c["beam_E_eV"] if c["beam_mode"] == 0 else (
            c["beam_Emin_eV"] + (c["beam_Emax_eV"] - c["beam_Emin_eV"]) * _u01(wv[1]))
        ub = torch.sqrt(2 * Eb * c["e"] / c["m_i"] + 0 * _u01(wv[1])) * self.dt / self.dx
        x = self.N - ub * _u01(wv[0])
        y = (c["beam_yc"] + c["beam_sigma"] * _normal(_u01(wv[2]), _u01(wv[3]))) / self.dy if self.ny else 0 * x
        y = y - self.ny * torch.floor(y / self.ny) if self.ny else y
        return [q.reshape(steps, B) for q in (x, -ub, y, 0 * x)]

    def run(self, steps):
        c, N = self.c, self.N
        base = int(self.ids.max()) + 1 if self.ids.numel() else 0
        self._solve(True, 0, 0.0, 0.0)
        B = int(c["beam_per_step"])
        beam = self._beam(steps) if B else None
        for n in range(steps):
            conv, energy, cfl, hits = 0, 0.0, 0.0, None
            for s in range(3):
                x, u, y, w = self.p[s]
                if not x.numel():
                    continue
                Ex, Ey = self._gather(x, y)
                f = (1.0 if self.pushed else 0.5) * self.charge[s] * c["e"] * self.dt ** 2 / self.mass[s]
                u = u + f / self.dx * Ex
                x = x + u
                cfl = max(cfl, float(u.abs().max()))
                if self.ny:
                    w = w + f / self.dy * Ey
                    y = torch.remainder(y + w, self.ny)
                    cfl = max(cfl, float(w.abs().max()))
                low, live = x <= 0, (x > 0) & (x < N)
                conv += self.charge[s] * int(low.sum())
                if s == 1:
                    gone = ~live
                    hits = (self.ids[gone], (~low[gone]).long(), u[gone], w[gone] if self.ny else 0 * u[gone],
                            y[gone] if self.ny else 0 * u[gone])
                    self.ids = self.ids[live]
                self.p[s] = [x[live], u[live], y[live] if self.ny else 0 * x[live],
                             w[live] if self.ny else 0 * x[live]]
            self.pushed = True
            if hits is not None and hits[0].numel():
                more, energy = self._emit(hits)
                conv += more
            if B:
                self._append(1, *(q[n] for q in beam))
                self.ids = torch.cat([self.ids, base + n * B + torch.arange(B, device=self.dev)])
            self.level += 1
            self._solve(False, conv, energy, cfl)


def _exact_run(case, seed, dev):
    cfg = _cfg(case, seed)
    sim = _Sim(cfg, case["mode"], dev)
    k = torch.arange(case["pairs"], device=dev)
    o = torch.zeros_like(k)
    wv = _philox(k, o, o, seed, 0x4C4F4144)
    x = cfg["n_cells"] * _u01(wv[0])
    if case["precision"] == "fp32":  # the store the plasma is drawn into
        x = x.float().clamp(1.2e-38, float(np.nextafter(np.float32(cfg["n_cells"]), np.float32(0)))).double()
    r, a = torch.sqrt(-2 * torch.log(_u01(wv[1]))), 2 * math.pi * _u01(wv[2])
    for s, z, m in ((0, r * torch.cos(a), cfg["m_e"]), (1, r * torch.sin(a), cfg["m_i"])):
        sim.p[s] = [x, W.thermal_u(cfg, m, cfg["T_load_eV"]) * z, 0 * x, 0 * x]
    sim.ids = k
    sim.run(case["steps"])
    rho = sim.G[:, 0].double() * (cfg["e"] * cfg["weight"] / (cfg["area"] * sim.dx * sim.fix))
    return dict(history=dict({k: np.array(v) for k, v in sim.rows.items()}, **{k: None for k in WHOLE}),
                grid=dict(phi=sim.phi, rho=rho, E=sim.E, G=None))


def _exact_2d(case, seed, dev):
    cfg = _cfg2d(case, seed)
    sim = _Sim(cfg, case["mode"], dev, ny=case["ny"])
    xi, eta, ue, we, ui, wi = (torch.from_numpy(v).to(dev) for v in W.load_pairs_2d(cfg))
    sim.p[0], sim.p[1] = [xi, ue, eta, we], [xi, ui, eta, wi]
    sim.ids = torch.arange(case["pairs"], device=dev)
    sim.run(case["steps"])
    hist = {k: np.array(v[1:]) for k, v in sim.rows.items()}  # level 0 is solved in prepare()
    return dict(history=dict(hist, **{k: None for k in WHOLE}), fields=dict(phi=sim.phi2, Ex=sim.Ex, Ey=sim.Ey, G=None))


def _exact_train(case, seed):
    X, Y, m, v = (q.double() for q in _train_inputs(case, seed))
    params = torch.empty(native.MLP_NPARAM, dtype=torch.float32, device="cuda")
    _ok(native.cp_mlp_init(params.data_ptr(), seed, native.current_stream()))
    p = params.double()
    # weights as the network holds them (bfloat16), biases as they are
    flat = p.clone()
    parts, at = [], 0
    for o, i in ((64, 40), (64, 64), (64, 64), (2, 64)):
        flat[at:at + o * i] = params[at:at + o * i].bfloat16().double()
        parts.append((at, o, i))
        at += o * i + o
    flat.requires_grad_(True)
    h = X
    for q, (at, o, i) in enumerate(parts):
        h = h @ flat[at:at + o * i].reshape(o, i).t() + flat[at + o * i:at + o * i + o]
        if q < 3:
            h = torch.nn.functional.gelu(h)
    loss = ((h - Y) ** 2).sum() / (2 * case["batch"])
    loss.backward()
    g = flat.grad
    b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
    m = b1 * m + (1 - b1) * g
    v = b2 * v + (1 - b2) * g * g
    p = p - float(np.float32(TRAIN_LR)) * (m / (1 - b1 ** TRAIN_T)) / (
        torch.sqrt(v / (1 - b2 ** TRAIN_T)) + float(np.float32(1e-8)))
    return dict(params=p, grad=g, loss=loss.detach().reshape(1), m=m, v=v)


def _exact_ions(case, seed):
    cfg, x, u, _, E = _ion_inputs(case, seed)
    N = case["cells"]
    x, u = x.double(), u.double()
    s = x - 0.5
    i = torch.floor(s).clamp(0, N - 1).long()
    t = torch.where(i >= N - 1, 0.0, (s - i).clamp(0, 1))
    f = E[i] + t * (E[(i + 1).clamp(max=N - 1)] - E[i])
    dx = cfg["d"] / N
    u = u + cfg["e"] * cfg["dt"] ** 2 / (cfg["m_i"] * dx) * f
    x = x + u
    live = (x > 0) & (x < N)
    return dict(xi=torch.where(live, x, -1.0), u=torch.where(live, u, 0.0), G=None, counts=None)


def exact(case, seed):
    kind = case["kind"]
    if kind == "run":
        return _exact_run(case, seed, torch.device("cuda"))
    if kind == "gap2d":
        return _exact_2d(case, seed, torch.device("cuda"))
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "ions":
        return _exact_ions(case, seed)
    return None  # hundreds to thousands of levels in: over 20 s, and the trajectories have long parted
