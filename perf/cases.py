"""Performance cases of the solver: what a user of this package has it do, through its public entry points.

Every case is one call (or one loop body) of a user's program on a state that a run meets in earnest:

* time steps of a simulation, with the state on the GPU (`Solver.step`, one pass = one SSP-RK3 step).  The states are
  mid-run states: shocks and material interfaces, waves of all strengths behind them down to round-off level, and
  undisturbed fluid ahead of them.  After RESTART steps the run begins again from its first state, so that a pass
  costs the same however often it is repeated;
* `ws_flux_divergence`, the semi-discrete operator, for programs with a time integrator of their own;
* `ws_run_host`, a step of a state in host memory (pinned), copies included;
* one training step of the learned gate (`ws_mlp_grad` and `ws_mlp_adam`).

Sizes are those of the package's workloads, tests and benchmark (200-cell tube, 96^2 and 1024^2 shock-bubble, 3000 x
1000 shock-cylinder, 256^3 drop, 4096 tubes, 65536 training faces) and ragged ones between them; `draw` covers the
ranges.  The outputs are the interior cells (ghost cells are scratch by the ABI's contract).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1707_00592_gb300 as ws
from paper_1707_00592_gb300 import learned

NG = 3
RESTART = 32        # steps of a run before it begins again
RESTART_HOST = 128  # the same for host-resident runs (the copy is the user's own and slow)

OPTS = {"precision": "mixed", "weights": "modified", "mood": True, "resident": False, "read_dt": False}


def listed():
    return [
        # the 200-cell gas-water shock tube, FP64, the program reading dt after each step to reach an end time: the
        # smallest call, latency and launches
        {"name": "tube_200_fp64", "kind": "step", "problem": "tube", "nx": 200, "ny": 1, "nz": 1, "precision": "fp64",
         "read_dt": True},
        # a resolved 1D tube in mixed precision, the same loop
        {"name": "tube_2000_mixed", "kind": "step", "problem": "tube", "nx": 2000, "ny": 1, "nz": 1, "read_dt": True},
        # a small 2D run, as for a parameter study: fewer tiles than SMs
        {"name": "bubble_96_mixed", "kind": "step", "problem": "bubble", "nx": 96, "ny": 96, "nz": 1},
        # the package's main workload: the shock-bubble in mixed precision, state owned by the run
        {"name": "bubble_1024_mixed", "kind": "step", "problem": "bubble", "nx": 1024, "ny": 1024, "nz": 1,
         "resident": True},
        # the largest 2D configuration: shock on a gas cylinder in a channel, reflective walls, MOOD off
        {"name": "cylinder_3000x1000_mixed", "kind": "step", "problem": "cylinder", "nx": 3000, "ny": 1000, "nz": 1,
         "mood": False},
        # the 3D configuration: a drop in periodic air with density noise everywhere
        {"name": "drop_256_mixed", "kind": "step", "problem": "drop", "nx": 256, "ny": 256, "nz": 256,
         "resident": True},
        # FP64 runs, the reference every mixed run is checked against: 2D and 3D
        {"name": "bubble_512_fp64", "kind": "step", "problem": "bubble", "nx": 512, "ny": 512, "nz": 1,
         "precision": "fp64"},
        {"name": "drop_48_fp64", "kind": "step", "problem": "drop", "nx": 48, "ny": 48, "nz": 48, "precision": "fp64"},
        # batched independent Riemann tubes of uneven length, per-tube time steps
        {"name": "tubes_4096_mixed", "kind": "tubes", "ntubes": 4096, "lmin": 256, "lmax": 8192},
        # the operator L(U) on a ragged grid with the comparison scheme's weights
        {"name": "flux_641x479_mixed_js", "kind": "flux", "problem": "bubble", "nx": 641, "ny": 479, "nz": 1,
         "weights": "js"},
        # a step of a host-resident state, copies included
        {"name": "host_1024_mixed", "kind": "host", "problem": "bubble", "nx": 1024, "ny": 1024, "nz": 1},
        # a training step of the face classifier: forward, backward, optimiser
        {"name": "train_65536", "kind": "train", "samples": 65536},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides(rng, cells, aspect=3.0, dims=2):
    """Ragged side lengths of about `cells` cells."""
    a = [math.exp(rng.uniform(-0.5, 0.5) * math.log(aspect)) for _ in range(dims)]
    scale = (cells / np.prod(a)) ** (1.0 / dims)
    return [max(8, int(v * scale)) for v in a]


def draw(rng):
    what = rng.choice(["tube", "grid2", "grid2", "grid2_fp64", "grid3", "grid3_fp64", "tubes", "tubes_fp64", "flux",
                       "host", "train"])
    weights = rng.choice(["modified", "modified", "modified", "basic", "js"])
    mood = rng.random() < 0.75
    if what == "tube":
        return {"kind": "step", "problem": "tube", "nx": _log_int(rng, 64, 20000), "ny": 1, "nz": 1,
                "precision": rng.choice(["fp64", "mixed"]), "weights": weights, "mood": mood, "read_dt": True}
    if what in ("grid2", "grid2_fp64"):
        fp64 = what == "grid2_fp64"
        nx, ny = _sides(rng, math.exp(rng.uniform(math.log(4000), math.log(2.4e5 if fp64 else 2.9e6))))
        return {"kind": "step", "problem": rng.choice(["bubble", "cylinder"]), "nx": nx, "ny": ny, "nz": 1,
                "precision": "fp64" if fp64 else "mixed", "weights": weights, "mood": mood,
                "resident": not fp64 and rng.random() < 0.5}
    if what in ("grid3", "grid3_fp64"):
        fp64 = what == "grid3_fp64"
        nx, ny, nz = _sides(rng, math.exp(rng.uniform(math.log(8000), math.log(1.0e5 if fp64 else 1.2e7))), 2.0, 3)
        return {"kind": "step", "problem": "drop", "nx": nx, "ny": ny, "nz": nz,
                "precision": "fp64" if fp64 else "mixed", "weights": weights, "mood": mood,
                "resident": not fp64 and rng.random() < 0.5}
    if what in ("tubes", "tubes_fp64"):
        fp64 = what == "tubes_fp64"
        lmax = _log_int(rng, 600, 4000 if fp64 else 8192)
        return {"kind": "tubes", "ntubes": _log_int(rng, 8, 64 if fp64 else 4096), "lmin": rng.randint(32, 256),
                "lmax": lmax, "precision": "fp64" if fp64 else "mixed", "weights": weights, "mood": mood}
    if what == "flux":
        fp64 = rng.random() < 0.5
        if rng.random() < 0.7:
            nx, ny = _sides(rng, math.exp(rng.uniform(math.log(4000), math.log(2e5 if fp64 else 1.2e6))))
            nz, problem = 1, rng.choice(["bubble", "cylinder"])
        else:
            nx, ny, nz = _sides(rng, math.exp(rng.uniform(math.log(8000), math.log(1e5 if fp64 else 1.2e6))), 2.0, 3)
            problem = "drop"
        return {"kind": "flux", "problem": problem, "nx": nx, "ny": ny, "nz": nz,
                "precision": "fp64" if fp64 else "mixed", "weights": weights, "mood": mood}
    if what == "host":
        nx, ny = _sides(rng, math.exp(rng.uniform(math.log(4e4), math.log(1e6))))
        return {"kind": "host", "problem": "bubble", "nx": nx, "ny": ny, "nz": 1, "weights": weights, "mood": mood}
    return {"kind": "train", "samples": _log_int(rng, 1000, 262144)}


# ---------------------------------------------------------------------------------------------------------------
# states
# ---------------------------------------------------------------------------------------------------------------
AIR, WATER = (1.4, 0.0), (4.4, 6.0e8)


def _opt(case, key):
    return case.get(key, OPTS.get(key))


def _pick(where, a, b):
    """a where the condition holds, b elsewhere, in 64 bits."""
    b = b if torch.is_tensor(b) else torch.full(where.shape, b, dtype=torch.float64, device=where.device)
    return torch.where(where, a, b)


def _material(gamma, pinf):
    return 1.0 / (gamma - 1.0), gamma * pinf / (gamma - 1.0)


def _waves(rng, coords, scale, count=5):
    """A smooth random field of unit size: `count` plane waves of wavelengths between scale and scale / 6."""
    s = 0.0
    for _ in range(count):
        k = rng.normal(size=len(coords))
        k = 2.0 * math.pi * k / np.linalg.norm(k) * rng.uniform(1.0, 6.0) / scale
        arg = rng.uniform(0.0, 2.0 * math.pi)
        for c, kc in zip(coords, k):
            arg = arg + float(kc) * c
        s = s + torch.sin(arg) / count
    return s


def _disturb(rng, coords, d, quiet, rho, vel, p, G, P, strength, reach, scale):
    """Acoustic and entropy waves around the fronts: d is the distance to the nearest shock or interface, over which
    their strength falls from `strength` to round-off level; none where `quiet` (fluid no wave has reached)."""
    env = strength * torch.exp(-d / reach) + 1e-3 * strength * torch.exp(-d / (4.0 * reach))
    env = torch.where(quiet, torch.zeros_like(env), env)
    rc2 = ((G + 1.0) * p + P) / G  # rho c^2
    c = torch.sqrt(rc2 / rho)
    a = env * _waves(rng, coords, scale)
    for k in range(len(vel)):
        vel[k] = vel[k] + (a if k == 0 else env * _waves(rng, coords, scale)) * c
    p = p + a * rc2
    rho = rho * (1.0 + a + 0.3 * env * _waves(rng, coords, scale))
    return rho, vel, p


def _axes(n, length, ndim):
    ax = [(torch.arange(n[d], dtype=torch.float64, device="cuda") + 0.5) * (length[d] / n[d]) for d in range(ndim)]
    if ndim == 1:
        return [ax[0]]
    return list(torch.meshgrid(*reversed(ax), indexing="ij"))[::-1]  # x, y(, z), each shaped (z, )y, x


def _fluid(case, seed):
    """(ndim, n, dx, bc, primitives): rho, velocities, p, Gamma, Pi of the interior cells, shaped (z, )y, x."""
    rng = np.random.default_rng([seed, 17])
    problem = case["problem"]
    n = (case["nx"], case["ny"], case["nz"])
    Gw, Pw = _material(*WATER)
    Ga, Pa = _material(*AIR)
    if problem == "tube":  # water under high pressure against air, and the fan and shock that have left the interface
        (X,) = _axes(n, (1.0,), 1)
        x0 = rng.uniform(0.6, 0.75)
        left, right = X < x0 - rng.uniform(0.05, 0.15), X >= x0 + rng.uniform(0.02, 0.05)
        water = X < x0
        G, P = _pick(water, Gw, Ga), _pick(water, Pw, Pa)
        rho = _pick(water, 900.0, rng.uniform(100.0, 200.0))
        p = torch.full_like(X, 1.0e6)
        rho = _pick(left, 1000.0, _pick(right, 50.0, rho))
        p = _pick(left, 1.0e9 * rng.uniform(0.8, 1.2), _pick(right, 1.0e5 * rng.uniform(0.8, 1.2), p))
        u = _pick(left | right, 0.0, rng.uniform(150.0, 250.0))
        d = torch.abs(X - x0)
        quiet = (X < 0.3) | (X > 0.9)
        rho, (u,), p = _disturb(rng, [X], d, quiet, rho, [u], p, G, P, 1e-2, 0.03, 0.1)
        return 1, n, (1.0 / n[0], 1.0, 1.0), (("transmissive", "transmissive"),), [rho, u, p, G, P]
    if problem == "bubble":  # a Ms = 1.5 water shock approaching an air bubble in water
        X, Y = _axes(n, (1.0, 1.0), 2)
        h = 1.0 / max(n[0], n[1])
        cx, cy, R = 0.55 + rng.uniform(-0.03, 0.03), 0.5 + rng.uniform(-0.05, 0.05), 0.2 * rng.uniform(0.9, 1.1)
        xs = cx + R + rng.uniform(0.01, 0.03)
        r = torch.hypot(X - cx, Y - cy)
        a = torch.clamp(0.5 + (R - r) / (2.0 * h), 0.0, 1.0)
        post = X > xs
        rho = _pick(post, 1259.07, a + (1.0 - a) * 1000.0)
        G, P = a * Ga + (1.0 - a) * Gw, a * Pa + (1.0 - a) * Pw
        u, v = _pick(post, -501.5, 0.0), torch.zeros_like(X)
        p = _pick(post, 1.2225e9, 1.0e5)
        quiet = X < rng.uniform(0.15, 0.25)
        d = torch.minimum(torch.abs(r - R), torch.abs(X - xs))
        rho, (u, v), p = _disturb(rng, [X, Y], d, quiet, rho, [u, v], p, G, P, 1e-2, 0.01, 0.3)
        bc = (("transmissive", "transmissive"), ("transmissive", "transmissive"))
        return 2, n, (1.0 / n[0], 1.0 / n[1], 1.0), bc, [rho, u, v, p, G, P]
    if problem == "cylinder":  # a Ms = 1.22 air shock and a cylinder of another gas in a channel with walls
        Lx, Ly = 0.267, 0.089
        X, Y = _axes(n, (Lx, Ly), 2)
        h = min(Lx / n[0], Ly / n[1])
        heavy = rng.random() < 0.5
        rho_in, g_in = (4.415, 1.249) if heavy else (0.255, 1.648)
        cx, cy, R = 0.15 + rng.uniform(-0.01, 0.01), 0.0445 + rng.uniform(-0.005, 0.005), 0.025 * rng.uniform(0.9, 1.1)
        xs = cx + R + rng.uniform(0.002, 0.01)
        r = torch.hypot(X - cx, Y - cy)
        a = torch.clamp(0.5 + (R - r) / (2.0 * h), 0.0, 1.0)
        post = X > xs
        rho = _pick(post, 1.927, a * rho_in + (1.0 - a) * 1.4)
        G, P = a * _material(g_in, 0.0)[0] + (1.0 - a) * Ga, torch.zeros_like(X)
        u, v = _pick(post, -114.42, 0.0), torch.zeros_like(X)
        p = _pick(post, 1.57e5, 1.0e5)
        quiet = X < rng.uniform(0.08, 0.11)
        d = torch.minimum(torch.abs(r - R), torch.abs(X - xs))
        rho, (u, v), p = _disturb(rng, [X, Y], d, quiet, rho, [u, v], p, G, P, 1e-2, 0.005, 0.08)
        bc = (("transmissive", "transmissive"), ("reflective", "reflective"))
        return 2, n, (Lx / n[0], Ly / n[1], 1.0), bc, [rho, u, v, p, G, P]
    # drop: water in periodic air, advected, density noise of 1 % everywhere
    X, Y, Z = _axes(n, (1.0, 1.0, 1.0), 3)
    h = 1.0 / max(n)
    c = [0.5 + rng.uniform(-0.05, 0.05) for _ in range(3)]
    r = torch.sqrt((X - c[0]) ** 2 + (Y - c[1]) ** 2 + (Z - c[2]) ** 2)
    a = torch.clamp(0.5 + (0.25 * rng.uniform(0.9, 1.1) - r) / (2.0 * h), 0.0, 1.0)
    S = torch.zeros_like(X)
    for _ in range(8):
        k = rng.integers(-4, 5, size=3)
        S += torch.sin(2.0 * math.pi * (float(k[0]) * X + float(k[1]) * Y + float(k[2]) * Z) + rng.uniform(0.0, 2.0 * math.pi))
    rho = (a * 1000.0 + (1.0 - a)) * (1.0 + 0.01 * S / torch.clamp(S.abs().max(), min=1e-30))
    vel = [torch.full_like(X, v) for v in (1.0, 0.5, 0.25)]
    bc = tuple(("periodic", "periodic") for _ in range(3))
    dx = tuple(1.0 / n[d] for d in range(3))
    return 3, n, dx, bc, [rho, *vel, torch.full_like(X, 1.0e5), a * Gw + (1.0 - a) * Ga, a * Pw + (1.0 - a) * Pa]


def _tubes(case, seed):
    """(offsets, primitives (5, cells)): Riemann problems in tubes of log-uniform length (the case's), each some time
    into its run (the waves from the midpoint have swept part of the tube)."""
    rng = np.random.default_rng([seed, 23])
    nt, lmin, lmax = case["ntubes"], case["lmin"], case["lmax"]
    spread = np.random.default_rng([nt, lmin, lmax]).uniform(math.log(lmin), math.log(lmax), size=nt)
    lens = np.clip(np.rint(np.exp(spread)).astype(np.int64), lmin, lmax)
    off = np.zeros(nt + 1, dtype=np.int64)
    off[1:] = np.cumsum(lens + 2 * NG)
    rho = np.exp(rng.uniform(0.0, math.log(1000.0), size=(2, nt)))
    p = np.exp(rng.uniform(math.log(1e5), math.log(1e9), size=(2, nt)))
    water = rng.integers(0, 2, size=(2, nt)).astype(bool)
    u = np.sort(rng.uniform(-100.0, 100.0, size=(2, nt)), axis=0)[::-1]  # approaching: no vacuum opens
    swept = rng.uniform(0.0, 500.0, size=nt)  # cells on either side of the midpoint
    gw, ga = np.array(_material(*WATER)), np.array(_material(*AIR))
    rows = np.concatenate([rho, u, p, np.where(water, gw[0], ga[0]), np.where(water, gw[1], ga[1])])  # (10, nt)
    rows = torch.from_numpy(np.ascontiguousarray(rows)).cuda()
    tube, lo, hi = _tube_index(off)
    at = torch.arange(int(off[-1]), device="cuda")
    at = torch.minimum(torch.maximum(at, lo), hi)  # ghost cells: the transmissive ends
    mid = lo + (hi + 1 - lo) // 2
    x = (at - mid).double()
    side = (at >= mid).long()
    q = [torch.gather(rows[2 * f:2 * f + 2][:, tube], 0, side[None])[0] for f in range(5)]
    d = torch.abs(x)
    quiet = d > torch.from_numpy(swept).cuda()[tube]
    r, (v,), pr = _disturb(rng, [x], d, quiet, q[0], [q[1]], q[2], q[3], q[4], 1e-2, 60.0, 60.0)
    return off, torch.stack([r, v, pr, q[3], q[4]])


def _tube_index(off):
    """Of every padded cell: its tube, and the first and last interior cell of that tube."""
    o = torch.from_numpy(off).cuda()
    tube = torch.repeat_interleave(torch.arange(len(off) - 1, device="cuda"), o[1:] - o[:-1])
    return tube, o[:-1][tube] + NG, o[1:][tube] - NG - 1


def _features(case, seed):
    """Training samples: normalised stencils of four characteristic variables and their labels."""
    rng = np.random.default_rng([seed, 29])
    g = torch.Generator(device="cuda")
    g.manual_seed(int(rng.integers(0, 2 ** 31)))
    n = case["samples"]
    w = torch.randn((n, 4, 6), generator=g, device="cuda", dtype=torch.float64).cumsum(2)
    flat = torch.rand((n, 4, 1), generator=g, device="cuda") < 0.3
    w = (w - w.mean(2, keepdim=True)) / (w.amax(2, keepdim=True) - w.amin(2, keepdim=True) + 1e-30)
    X = torch.where(flat, torch.zeros_like(w), w).reshape(n, 24).float().contiguous()
    y = (torch.rand(n, generator=g, device="cuda") < 0.25).to(torch.uint8)
    return X, y, learned.init_params(int(rng.integers(0, 2 ** 31)))


# ---------------------------------------------------------------------------------------------------------------
# what the user has in hand, and one pass
# ---------------------------------------------------------------------------------------------------------------
def _inner(s, t):
    """The interior cells of a state buffer."""
    sl = [slice(None)] + [slice(NG, NG + s.n[d]) if d < s.ndim else slice(None) for d in (2, 1, 0)]
    return t[tuple(sl)]


def _solver(case, seed):
    ndim, n, dx, bc, prim = _fluid(case, seed)
    s = ws.Solver(ndim, n, dx, bc, precision=_opt(case, "precision"), weights=_opt(case, "weights"),
                  mood=_opt(case, "mood"))
    Q = s.tensor()
    _inner(s, Q).copy_(torch.stack(prim).reshape(_inner(s, Q).shape))
    return s, s.prim_to_cons(Q)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        X, y, P = _features(case, seed)
        P = torch.tensor(P, dtype=torch.float32, device="cuda")
        return {"kind": kind, "X": X, "y": y, "P": P, "M": torch.zeros_like(P), "V": torch.zeros_like(P),
                "G": torch.empty_like(P), "L": torch.empty(1, dtype=torch.float32, device="cuda"), "n": 0}
    if kind == "tubes":
        off, Q = _tubes(case, seed)
        s = ws.Solver(1, (1, 1, 1), (1.0, 1.0, 1.0), None, tube_offsets=off, precision=_opt(case, "precision"),
                      weights=_opt(case, "weights"), mood=_opt(case, "mood"))
        U = s.prim_to_cons(Q.contiguous())
        return {"kind": kind, "s": s, "U": U, "U0": U.clone(), "n": 0}
    s, U = _solver(case, seed)
    if kind == "flux":
        return {"kind": kind, "s": s, "U": U, "L": s.tensor()}
    if kind == "host":
        U0 = U.cpu()
        Uh = torch.empty(U0.shape, dtype=torch.float64, pin_memory=True)
        Uh.copy_(U0)
        return {"kind": kind, "s": s, "U": Uh, "U0": U0, "n": 0}
    if _opt(case, "resident"):
        ws.ws_set_resident(s.ctx, True)
    return {"kind": kind, "s": s, "U": U, "U0": U.clone(), "n": 0, "resident": _opt(case, "resident"),
            "read_dt": _opt(case, "read_dt")}


def run(state):
    kind = state["kind"]
    if kind == "train":
        state["n"] += 1
        ws.ws_mlp_grad(state["P"], state["X"], state["y"], 3.0, state["G"], state["L"])
        ws.ws_mlp_adam(state["P"], state["M"], state["V"], state["G"], state["n"], 3e-3)
        return {k: state[k] for k in ("P", "M", "V", "G", "L")}
    s, U = state["s"], state["U"]
    if kind == "flux":
        ws.ws_flux_divergence(s.ctx, U, state["L"])
        return _inner(s, state["L"])
    if state["n"] == (RESTART_HOST if kind == "host" else RESTART):  # the run begins again
        U.copy_(state["U0"])
        if state.get("resident"):
            ws.ws_set_resident(s.ctx, True)  # the state was changed outside the solver
        state["n"] = 0
    state["n"] += 1
    if kind == "host":
        ws.ws_run_host(s.ctx, U, 1)
        return _inner(s, U)
    if kind == "tubes":
        s.step(U)
        return U  # the tubes lie one after another, their ghost cells (those of the first state) between them
    if state["read_dt"]:
        dt = s.step(U, want_dt=True)
        return {"U": _inner(s, U), "dt": dt}
    s.step(U)
    return _inner(s, U)


def _cells(case):
    if case["kind"] != "tubes":
        return case["nx"] * case["ny"] * case["nz"]
    mean = (case["lmax"] - case["lmin"]) / math.log(case["lmax"] / case["lmin"])
    return int(case["ntubes"] * mean)


def work(case):
    """One pass: the state read and written once; the method's operations per face and cell (an addition, product,
    division, root or comparison each counts as one)."""
    if case["kind"] == "train":
        n, weights = case["samples"], 24 * 32 + 32 * 32 + 32
        return {"bytes": n * (24 * 4 + 1) + 8 * 4 * 1889, "flops": 6 * n * weights}
    ndim = {"tube": 1, "bubble": 2, "cylinder": 2, "drop": 3}[case["problem"]] if case["kind"] != "tubes" else 1
    cells, nv = _cells(case), ndim + 4
    per_stage = cells * (ndim * {1: 1251, 2: 1469, 3: 1687}[ndim] + {1: 31, 2: 62, 3: 99}[ndim])
    return {"bytes": 16 * nv * cells, "flops": (1 if case["kind"] == "flux" else 3) * per_stage}


# ---------------------------------------------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------------------------------------------
def _sound2(rho, p, G, P):
    return ((G + 1.0) * p + P) / (G * rho)


def _prim(U, ndim):
    rho, m = U[0], U[1:1 + ndim]
    vel = [c / rho for c in m]
    ke = 0.5 * rho * sum(v * v for v in vel)
    E, G, P = U[1 + ndim:4 + ndim]
    p = ((E - ke) - P) / G
    return [rho, *vel, p, G, P]


def _weno(v, order, weights, mixed):
    """Left value at i+1/2 from the cells i-2..i+2."""
    a, b, c, d, e = v  # q_{i-2} .. q_{i+2}
    k = 13.0 / 12.0
    d1, d2 = 0.5 * (d - c), 0.5 * (c - b)
    d3 = (5.0 / 6.0) * (d - c) - (1.0 / 6.0) * (e - c)
    d4 = (1.0 / 3.0) * (a - c) - (7.0 / 6.0) * (b - c)
    b12 = k * (b - 2.0 * c + d) ** 2 + 0.25 * (b - d) ** 2
    b3 = k * (c - 2.0 * d + e) ** 2 + 0.25 * (3.0 * c - 4.0 * d + e) ** 2
    b4 = k * (a - 2.0 * b + c) ** 2 + 0.25 * (a - 4.0 * b + 3.0 * c) ** 2
    if weights == "js" and order == 5:
        dc = (1.0 / 3.0) * (d - c) - (1.0 / 6.0) * (b - c)
        a0, a1, a2 = 1.0 / (1e-6 + b4) ** 2, 6.0 / (1e-6 + b12) ** 2, 3.0 / (1e-6 + b3) ** 2
        return c + (a0 * d4 + a1 * dc + a2 * d3) / (a0 + a1 + a2)
    b1, b2 = (d - c) ** 2, (c - b) ** 2
    tau = 0.25 * (e - 2.0 * d + 2.0 * b - a) ** 2 + k * (e - 4.0 * d + 6.0 * c - 4.0 * b + a) ** 2
    eps = 1e-10 * (b1 + b2 + tau) + 1e-30 if mixed else 1e-40
    r1, r2 = tau / (b1 + eps), tau / (b2 + eps)
    if weights != "basic":
        r12 = tau / (b12 + eps)
        r1, r2 = r1 * r12, r2 * r12
    a1, a2 = 4.0 * (1.0 + r1), 2.0 * (1.0 + r2)
    num, den = a1 * d1 + a2 * d2, a1 + a2
    if order == 5:
        a3, a4 = 3.0 * (1.0 + tau / (b3 + eps)), 1.0 + tau / (b4 + eps)
        num, den = num + a3 * d3 + a4 * d4, den + a3 + a4
    return c + num / den


def _states(q, c, weights, mood, mixed):
    """Both states of every face from the sweep-frame primitives (rho, u_n, u_t.., p, Gamma, Pi) of its six cells."""
    nq = len(q[0])
    ip = nq - 3
    rb, cb = 0.5 * (q[2][0] + q[3][0]), 0.5 * (c[2] + c[3])
    rc, c2 = rb * cb, cb * cb

    def project(k, r):
        if r == 0:
            return -0.5 * rc * q[k][1] + 0.5 * q[k][ip]
        if r == 1:
            return q[k][0] - q[k][ip] / c2
        if r == nq - 1:
            return 0.5 * rc * q[k][1] + 0.5 * q[k][ip]
        return q[k][r] if r < ip else q[k][r + 1]

    def side(cells, order):
        w = []
        for r in range(nq):
            w.append(_weno([project(k, r) for k in cells], order, weights if order == 5 or weights != "js" else "modified",
                           mixed))
        return [(w[0] + w[-1]) / c2 + w[1], (w[-1] - w[0]) / rc, *w[2:ip], w[0] + w[-1], w[ip], w[ip + 1]]

    def fine(s):
        return (s[0] > 0) & (s[ip + 1] > 0) & ((s[ip + 1] + 1.0) * s[ip] + s[ip + 2] > 0)

    out = []
    for cells, own in (((0, 1, 2, 3, 4), 2), ((5, 4, 3, 2, 1), 3)):
        s = side(cells, 5)
        if mood and not bool(fine(s).all()):
            low = side(cells, 3)
            ok5, ok3 = fine(s), fine(low)
            s = [torch.where(ok5, x, torch.where(ok3, y, z)) for x, y, z in zip(s, low, q[own])]
        out.append(s)
    return out


def _hllc(l, r):
    nq = len(l)
    ip = nq - 3
    sides = []
    for s in (l, r):
        rho, un, p, G, P = s[0], s[1], s[ip], s[ip + 1], s[ip + 2]
        E = G * p + P + 0.5 * rho * sum(v * v for v in s[1:ip])
        U = [rho, rho * un, *[rho * t for t in s[2:ip]], E, G, P]
        F = [rho * un, rho * un * un + p, *[rho * un * t for t in s[2:ip]], (E + p) * un, G * un, P * un]
        sides.append((U, F, _sound2(rho, p, G, P)))
    sl, sr = torch.sqrt(l[0]), torch.sqrt(r[0])
    den = sl + sr
    ub = (sl * l[1] + sr * r[1]) / den
    cb = torch.sqrt((sl * sides[0][2] + sr * sides[1][2]) / den + 0.5 * sl * sr / (den * den) * (r[1] - l[1]) ** 2)
    Sl = torch.clamp(torch.minimum(ub - cb, l[1] - torch.sqrt(sides[0][2])), max=0.0)
    Sr = torch.clamp(torch.maximum(ub + cb, r[1] + torch.sqrt(sides[1][2])), min=0.0)
    ml, mr = l[0] * (Sl - l[1]), r[0] * (Sr - r[1])
    Ss = (r[ip] - l[ip] + ml * l[1] - mr * r[1]) / (ml - mr)
    left = 0.5 * (1.0 + torch.sign(Ss))
    flux, us = [], 0.0
    for (U, F, _), s, S, w in ((sides[0], l, Sl, left), (sides[1], r, Sr, 1.0 - left)):
        same = S == Ss
        dS = torch.where(same, torch.ones_like(S), S - Ss)
        Pk = s[ip] + s[0] * (S - s[1]) * (Ss - s[1])
        for m in range(nq):
            t = Ss * (S * U[m] - F[m])
            if m == 1:
                t = t + S * Pk
            if m == ip:
                t = t + S * Pk * Ss
            f = w * torch.where(same, F[m], t / dS)
            if len(flux) <= m:
                flux.append(f)
            else:
                flux[m] = flux[m] + f
        us = us + w * torch.where(same, s[1], Ss * (S - s[1]) / dS)
    return flux, us


def _ghosts(f, axis, kinds, flip):
    n = f.shape[axis]
    ends = []
    for end, kind in enumerate(kinds):
        if kind == "periodic":
            g = f.narrow(axis, n - NG, NG) if end == 0 else f.narrow(axis, 0, NG)
        elif kind == "reflective":
            g = (f.narrow(axis, 0, NG) if end == 0 else f.narrow(axis, n - NG, NG)).flip(axis)
            g = -g if flip else g
        else:
            shape = list(f.shape)
            shape[axis] = NG
            g = f.narrow(axis, 0 if end == 0 else n - 1, 1).expand(shape)
        ends.append(g)
    return torch.cat([ends[0], f, ends[1]], axis)


def _rhs(U, ndim, dx, bc, weights, mood, mixed):
    """L(U) of the interior cells U (nv, (z, )y, x)."""
    Q = _prim(U, ndim)
    L = [torch.zeros_like(f) for f in Q]
    for d in range(ndim):
        axis = U.dim() - 2 - d
        n = Q[0].shape[axis]
        order = [0, 1 + d] + [1 + e for e in range(ndim) if e != d] + [1 + ndim, 2 + ndim, 3 + ndim]
        pad = [_ghosts(Q[m], axis, bc[d], m == 1 + d) for m in order]
        cs = torch.sqrt(_sound2(pad[0], pad[-3], pad[-2], pad[-1]))
        q = [[f.narrow(axis, k, n + 1) for f in pad] for k in range(6)]
        c = [cs.narrow(axis, k, n + 1) for k in range(6)]
        l, r = _states(q, c, weights, mood, mixed)
        F, us = _hllc(l, r)
        for m, f in zip(order, F):
            L[m] = L[m] - (f.narrow(axis, 1, n) - f.narrow(axis, 0, n)) / dx[d]
        du = (us.narrow(axis, 1, n) - us.narrow(axis, 0, n)) / dx[d]
        for m in (2 + ndim, 3 + ndim):
            L[m] = L[m] + U[m] * du
        del pad, cs, q, c, l, r, F, us
    return torch.stack(L)


def _tubes_rhs(U, left, index, dx, weights, mood, mixed):
    """L(U) of concatenated tubes: face i+1/2 stored at cell i; index[k]: the cell i-2+k within its tube's ends."""
    Q = _prim(U, 1)
    cs = torch.sqrt(_sound2(Q[0], Q[2], Q[3], Q[4]))
    l, r = _states([[f[ix] for f in Q] for ix in index], [cs[ix] for ix in index], weights, mood, mixed)
    F, us = _hllc(l, r)
    L = torch.stack([-(f - f[left]) / dx for f in F])
    L[3:] += U[3:] * ((us - us[left]) / dx)
    return L


def _step(U, rhs, dt):
    U1 = U + dt * rhs(U)
    U2 = 0.75 * U + 0.25 * (U1 + dt * rhs(U1))
    return U / 3.0 + (2.0 / 3.0) * (U2 + dt * rhs(U2))


def _exact_train(case, seed):
    X, y, P = _features(case, seed)
    P = torch.tensor(P, dtype=torch.float32, device="cuda").double().requires_grad_(True)
    parts, at = [], 0
    for shape in ((32, 24), (32,), (32, 32), (32,), (32,), (1,)):
        size = math.prod(shape)
        parts.append(P[at:at + size].reshape(shape))
        at += size
    W1, b1, W2, b2, W3, b3 = parts
    h = torch.relu(torch.relu(X.double() @ W1.T + b1) @ W2.T + b2)
    z = h @ W3 + b3
    loss = torch.nn.functional.binary_cross_entropy_with_logits(z, y.double(), pos_weight=torch.tensor(3.0, dtype=torch.float64, device="cuda"))
    (G,) = torch.autograd.grad(loss, P)
    P = P.detach()
    return {"P": P - 3e-3 * G / (G.abs() + 1e-8), "M": 0.1 * G, "V": 1e-3 * G * G, "G": G, "L": loss.detach()[None]}


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    weights, mood, mixed = _opt(case, "weights"), _opt(case, "mood"), _opt(case, "precision") == "mixed"
    if kind == "tubes":
        off, Q = _tubes(case, seed)
        rho, u, p, G, P = Q
        U = torch.stack([rho, rho * u, G * p + P + 0.5 * rho * u * u, G, P])
        tube, lo, hi = _tube_index(off)
        at = torch.arange(U.shape[1], device="cuda")
        inner = (at >= lo) & (at <= hi)
        # transmissive ends: every stencil cell is brought inside its tube
        index = [torch.minimum(torch.maximum(at + k - 2, lo), hi) for k in range(6)]
        left = torch.clamp(at - 1, min=0)
        dx = 1.0 / (hi + 1 - lo).double()
        q = _prim(U, 1)
        rate = torch.where(inner, (q[1].abs() + torch.sqrt(_sound2(q[0], q[2], q[3], q[4]))) / dx, 0.0)
        top = torch.zeros(len(off) - 1, dtype=torch.float64, device="cuda").scatter_reduce(0, tube, rate, "amax")
        dt = (0.5 / top)[tube]
        new = _step(U, lambda V: _tubes_rhs(V, left, index, dx, weights, mood, mixed), dt)
        return torch.where(inner, new, U)
    ndim, n, dx, bc, prim = _fluid(case, seed)
    G, P = prim[-2:]
    U = torch.stack([prim[0], *[prim[0] * v for v in prim[1:1 + ndim]],
                     G * prim[1 + ndim] + P + 0.5 * prim[0] * sum(v * v for v in prim[1:1 + ndim]), G, P])

    def rhs(V):
        return _rhs(V, ndim, dx, bc, weights, mood, mixed)

    shape = (ndim + 4, *(n[d] if d < ndim else 1 for d in (2, 1, 0)))
    if kind == "flux":
        return rhs(U).reshape(shape)
    q = _prim(U, ndim)
    c = torch.sqrt(_sound2(q[0], *q[-3:]))
    dt = 0.5 / sum((q[1 + d].abs() + c) / dx[d] for d in range(ndim)).max()
    new = _step(U, rhs, dt).reshape(shape)
    if _opt(case, "read_dt"):
        return {"U": new, "dt": float(dt)}
    return new.cpu() if kind == "host" else new
