"""Performance cases of the hydro framework: what a user's program has it do.

The calls are the ones a simulation driver makes: whole RK3 steps of a uniform
octree level (``UniformRun``'s descriptor), whole RK3 steps of an adaptive
octree (``AMRRun``'s), one stage of a batch of leaf sub-grids
(``hydro_step`` and its allocation-free form), and the learned indicator's
training data and training steps.  A time step always advances buffer a into
buffer b (parity 0), so that every pass starts from the same state.

``exact`` is the method in plain torch FP64: PPM on the 13 lines through a
cell, Kurganov-Tadmor fluxes at the 9 points of a face, Simpson sums, sources,
SSP-RK3, ghost fill and flux correction.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2107_10987_gb300 import amr as A
from paper_2107_10987_gb300 import hydro as H
from paper_2107_10987_gb300 import workloads as W
from paper_2107_10987_gb300.uniform import UniformRun

DEV = "cuda"
F64 = torch.float64
GAMMA = 5.0 / 3.0
NF = 10
G = 3
ETA1, ETA2 = 1e-3, 0.1
FLOWS = ("blast", "star")


# ---------------------------------------------------------------------------
# the cases

def _uniform(name, nb, prec, fused, flow="blast", N=8, bc="outflow", points=9, contact=False, spin=False,
             indicator=False):
    c = dict(kind="uniform", nbx=nb[0], nby=nb[1], nbz=nb[2], precision=prec, fused=fused, flow=flow, N=N, bc=bc,
             points=points, contact=contact, spin=spin, indicator=indicator)
    return dict(c, name=name) if name else c


def _amr(name, leaves, lmin, lmax, prec):
    c = dict(kind="amr", leaves=leaves, lmin=lmin, lmax=lmax, precision=prec)
    return dict(c, name=name) if name else c


def _batch(name, n, prec, contact, spin, faces, static=False, N=8):
    c = dict(kind="batch", n=n, precision=prec, contact=contact, spin=spin, faces=faces, static=static, N=N)
    return dict(c, name=name) if name else c


def listed():
    return [
        # one 8^3 sub-grid with periodic ghosts in plain FP64: the smallest call, the first thing anyone runs
        _uniform("sedov_1_fp64", (1, 1, 1), "fp64", False, bc="periodic"),
        # the 64^3 blast of 512 sub-grids, in the fused mixed form and in plain FP64 (the accuracy reference)
        _uniform("blast_512_mixed_fused", (8, 8, 8), "mixed", True),
        _uniform("blast_512_fp64", (8, 8, 8), "fp64", False),
        # the same with the learned smoothness indicator on
        _uniform("blast_512_indicator", (8, 8, 8), "mixed", True, indicator=True),
        # the rotating star with gravity on 32,768 sub-grids (256^3): the largest single-GPU mesh, the headline
        _uniform("star_32768_mixed_fused", (32, 32, 32), "mixed", True, flow="star"),
        # 128^3 as 512 sub-grids of 16^3, as separate launches (the default of UniformRun)
        _uniform("star_512_n16_mixed", (8, 8, 8), "mixed", False, flow="star", N=16),
        # the old hydro module (face centres only) on a ragged mesh, FP64: the accuracy comparison runs
        _uniform("old_module_105_fp64", (5, 3, 7), "fp64", False, flow="star", points=1, bc="periodic"),
        # an adaptive octree around a blast shell, about 4,000 leaves at levels 3..6, mixed: the production run
        _amr("shell_4040_mixed", 4096, 3, 6, "mixed"),
        # a smaller adaptive octree in plain FP64
        _amr("shell_700_fp64", 700, 2, 5, "fp64"),
        # one stage of a ragged batch of leaves with contact steepening, spin feedback and boundary-face sums
        _batch("stage_77_contact_spin", 77, "mixed", True, True, True),
        # the indicator: features and labels of a snapshot's cells, and their predictions
        dict(kind="labels", name="labels_512", n=512),
        # the indicator: one training step at the driver's default minibatch
        dict(kind="train", name="train_65536", n=65536),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["uniform"] * 5 + ["amr", "amr", "batch", "batch", "labels", "train"])
    if kind == "uniform":
        prec = rng.choice(["mixed", "mixed", "fp64"])
        N = rng.choice([8, 8, 8, 16])
        # FP64 steps cost about 17 times the mixed ones: fewer sub-grids
        most = (20000 if prec == "mixed" else 1000) // (N // 8) ** 3
        n = _log_int(rng, 1, most)
        nbx = max(1, min(n, int(round(n ** (1 / 3) * rng.uniform(0.6, 1.7)))))
        nby = max(1, min(n // nbx, int(round((n / nbx) ** 0.5 * rng.uniform(0.6, 1.7)))))
        nbz = max(1, n // (nbx * nby))
        ind = rng.random() < 0.15
        return _uniform(None, (nbx, nby, nbz), prec, prec == "mixed" and rng.random() < 0.7, rng.choice(FLOWS), N,
                        rng.choice(["outflow", "periodic"]), rng.choice([9, 9, 9, 9, 1]),
                        not ind and rng.random() < 0.2, not ind and rng.random() < 0.15, ind)
    if kind == "amr":
        lmin = rng.choice([2, 3])
        lmax = lmin + rng.choice([1, 2, 3])
        prec = rng.choice(["mixed", "mixed", "fp64"])
        return _amr(None, _log_int(rng, max(100, 8 ** lmin), 4096 if prec == "mixed" else 1000), lmin, lmax, prec)
    if kind == "batch":
        prec = rng.choice(["mixed", "fp64"])
        static = prec == "fp64" and rng.random() < 0.5
        n = _log_int(rng, 1, H.HYDRO_STATIC_MAX_SUB if static else 4096 if prec == "mixed" else 1000)
        return _batch(None, n, prec, rng.random() < 0.5, not static and rng.random() < 0.5,
                      not static and rng.random() < 0.5, static)
    if kind == "labels":
        return dict(kind="labels", n=_log_int(rng, 8, 2048))
    return dict(kind="train", n=_log_int(rng, 4096, 131072))


# ---------------------------------------------------------------------------
# states: cell averages on the GPU, made from the seed alone

def _conserved(rho, v, p, z, frac):
    eps = p / (GAMMA - 1.0)
    U = torch.empty((rho.shape[0], NF) + rho.shape[1:], dtype=F64, device=rho.device)
    U[:, 0] = rho
    U[:, 1:4] = rho.unsqueeze(1) * v
    U[:, 4] = eps + 0.5 * rho * (v * v).sum(1)
    U[:, 5] = eps ** (1.0 / GAMMA)
    U[:, 6:9] = z
    U[:, 9] = rho * frac
    return U


def _blast(X, Y, Z, q):
    """A blast shell: gas at rest outside, a self-similar-like profile inside."""
    dx, dy, dz = X - q["c"][0], Y - q["c"][1], Z - q["c"][2]
    r = torch.sqrt(dx * dx + dy * dy + dz * dz)
    R = q["R"]
    inside = r < R
    jump = (GAMMA + 1.0) / (GAMMA - 1.0)
    rho = torch.where(inside, (jump * (r / R) ** (3.0 / (GAMMA - 1.0))).clamp_min(1e-3), torch.ones_like(r))
    vr = torch.where(inside, 0.75 * r / R, torch.zeros_like(r)) / r.clamp_min(1e-12)
    wob = 1.0 + 0.05 * torch.sin(q["k"][0] * X + q["ph"][0]) * torch.sin(q["k"][1] * Y + q["ph"][1])
    v = torch.stack([vr * dx * wob, vr * dy, vr * dz], 1)
    p = torch.where(inside, 0.3 + 0.45 * (r / R) ** 2, torch.full_like(r, 1e-5))
    z = torch.stack([torch.where(inside, 1e-3 * torch.sin(q["k"][m] * Z + q["ph"][m]), torch.zeros_like(r))
                     for m in range(3)], 1)
    frac = torch.where(inside, 0.5 + 0.2 * torch.sin(q["k"][2] * X + q["ph"][2]), torch.ones_like(r))
    return _conserved(rho, v, p, z, frac), None


@functools.lru_cache(maxsize=1)
def _polytrope():
    return W.polytrope_model(1.5, 0.5)


def _star(X, Y, Z, q):
    """A rotating n = 1.5 polytrope in a thin ambient medium, with its static gravity; a few percent of noise."""
    mo = _polytrope()
    r = torch.sqrt(X * X + Y * Y + Z * Z)
    tab = {k: torch.tensor(mo[k], dtype=F64, device=X.device) for k in ("xi", "theta", "m")}
    xi = r / mo["alpha"]
    i = torch.searchsorted(tab["xi"], xi.reshape(-1)).clamp(1, len(mo["xi"]) - 1).reshape(xi.shape)
    f = ((xi - tab["xi"][i - 1]) / (tab["xi"][i] - tab["xi"][i - 1])).clamp(0.0, 1.0)
    th = (tab["theta"][i - 1] * (1 - f) + tab["theta"][i] * f).clamp_min(0.0)
    m = tab["m"][i - 1] * (1 - f) + tab["m"][i] * f
    rho = (mo["rho_c"] * th ** mo["n"]).clamp_min(1e-10)
    p = mo["K"] * rho ** (1.0 + 1.0 / mo["n"])
    noise = 1.0 + 0.02 * torch.sin(q["k"][0] * X + q["ph"][0]) * torch.cos(q["k"][1] * Y + q["ph"][1])
    w = q["spin"] * mo["omega_K"]
    inside = (r < mo["R"]).to(F64)
    vs = 0.01 * torch.sin(q["k"][2] * Z + q["ph"][2])
    v = torch.stack([inside * (-w * Y + vs), inside * (w * X - vs), inside * vs], 1)
    z = torch.zeros_like(v)
    fg = torch.where(r > 0.0, -4.0 * math.pi * mo["alpha"] ** 3 * mo["rho_c"] * mo["G"] * m / r.clamp_min(1e-12) ** 3,
                     torch.zeros_like(r))
    g = torch.stack([fg * X, fg * Y, fg * Z], 1)
    return _conserved(rho * noise, v, p * noise, z, 0.5 + 0.3 * (noise - 1.0) / 0.02), g


def _params(seed):
    rng = np.random.default_rng(seed)
    return dict(c=rng.uniform(-0.1, 0.1, 3), R=rng.uniform(0.25, 0.4), k=rng.uniform(5.0, 40.0, 3),
                ph=rng.uniform(0.0, 2 * math.pi, 3), spin=rng.uniform(0.15, 0.25))


def _centres(origin, h, N):
    """Cell centres [n][N][N][N] of every sub-grid."""
    i = torch.arange(N, dtype=F64, device=origin.device) + 0.5
    hh = h.view(-1, 1, 1, 1)
    X = origin[:, 0].view(-1, 1, 1, 1) + hh * i.view(1, 1, 1, N)
    Y = origin[:, 1].view(-1, 1, 1, 1) + hh * i.view(1, 1, N, 1)
    Z = origin[:, 2].view(-1, 1, 1, 1) + hh * i.view(1, N, 1, 1)
    return torch.broadcast_tensors(X, Y, Z)


def _state(flow, origin, h, N, q):
    """Interiors [n][F][N][N][N] and gravity (or None), in chunks of the batch."""
    n = origin.shape[0]
    U = torch.empty((n, NF, N, N, N), dtype=F64, device=DEV)
    g = torch.empty((n, 3, N, N, N), dtype=F64, device=DEV) if flow == "star" else None
    chunk = max(1, 4096 // (N // 8) ** 3)
    for a in range(0, n, chunk):
        X, Y, Z = _centres(origin[a:a + chunk], h[a:a + chunk], N)
        u, gg = (_star if flow == "star" else _blast)(X, Y, Z, q)
        U[a:a + chunk] = u
        if g is not None:
            g[a:a + chunk] = gg
    return U, g


def _mesh(case):
    """Origins and cell width of a uniform level around the centre of [-1, 1]^3."""
    N = case["N"]
    nx, ny, nz = case["nbx"], case["nby"], case["nbz"]
    h = 2.0 / (N * max(nx, ny, nz))
    s = torch.arange(nx * ny * nz, device=DEV)
    k = torch.stack([s % nx, (s // nx) % ny, s // (nx * ny)], 1).to(F64)
    half = torch.tensor([nx, ny, nz], dtype=F64, device=DEV) / 2
    origin = (k - half) * (N * h)
    return origin, torch.full((nx * ny * nz,), h, dtype=F64, device=DEV)


def _indicator(seed):
    """Network parameters of the kind that training gives: the output grows with the relative differences in a
    cell's 3x3x3 block, so that cells in a uniform neighbourhood are the smooth ones."""
    rng = np.random.default_rng(seed + 77)
    W1 = rng.normal(0.0, 1.0, (32, 54))
    b1 = rng.uniform(-0.01, 0.01, 32)
    W2 = np.abs(rng.normal(0.0, 0.4, (32, 32)))
    b2 = rng.uniform(-0.01, 0.01, 32)
    w3 = np.abs(rng.normal(0.0, 0.4, 32))
    return torch.tensor(np.concatenate([W1.ravel(), b1, W2.ravel(), b2, w3, [-5.0]]), dtype=torch.float32, device=DEV)


def _context(case, omega=0.0):
    ctx = H.Context(GAMMA, omega, N=case.get("N", 8))
    prec = H.HYDRO_PREC_MIXED if case["precision"] == "mixed" else H.HYDRO_PREC_FP64
    H.hydro_set_mode(ctx, prec, 0.4, ETA1, ETA2, case.get("points", 9), int(case.get("contact", False)),
                     int(case.get("spin", False)))
    return ctx


def _omega(case, q):
    return q["spin"] if case.get("flow") == "star" else 0.0


def _bc(case):
    return H.HYDRO_BC_PERIODIC if case["bc"] == "periodic" else H.HYDRO_BC_OUTFLOW


@functools.lru_cache(maxsize=8)
def _leaves(target, lmin, lmax):
    level, ijk, _ = W.amr_shell_mesh(target, 1234, lmin, lmax)
    return level, ijk


def _amr_mesh(case, seed):
    level, ijk = _leaves(case["leaves"], case["lmin"], case["lmax"])
    perm = np.random.default_rng(seed).permutation(len(level))
    return level[perm], ijk[perm]


def _random_batch(case, seed):
    """Ghost-padded leaves full of contacts: two density levels with noise, small pressure noise, every fourth with
    a pressure jump."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    n, S = case["n"], case["N"] + 2 * G
    sh = (n, S, S, S)

    def uni(lo, hi, s=sh):
        return lo + (hi - lo) * torch.rand(s, generator=gen, dtype=F64, device=DEV)

    rho = torch.where(uni(0, 1) < 0.5, torch.ones(sh, dtype=F64, device=DEV),
                      torch.full(sh, 0.3, dtype=F64, device=DEV)) * uni(0.95, 1.05)
    p = uni(0.98, 1.02)
    p[3::4, :, :, : S // 2] *= 10.0
    v = uni(-0.3, 0.3, (n, 3, S, S, S))
    z = uni(-0.01, 0.01, (n, 3, S, S, S))
    U = _conserved(rho, v, p, z, uni(0.4, 0.6))
    origin = uni(-1.0, 1.0, (n, 3))
    h = 2.0 / (case["N"] * 2.0 ** torch.randint(3, 7, (n,), generator=gen, device=DEV).to(F64))
    return U, origin, h


def _snapshot(case, seed):
    """Ghost-filled sub-grids of a blast's mesh, as the indicator's training data sees them."""
    n = case["n"]
    nb = max(1, int(math.ceil(n ** (1 / 3))))
    h0 = 2.0 / (8 * nb)
    s = torch.arange(n, device=DEV)
    k = torch.stack([s % nb, (s // nb) % nb, s // (nb * nb)], 1).to(F64)
    origin = -1.0 + k * (8 * h0)
    h = torch.full((n,), h0, dtype=F64, device=DEV)
    q = _params(seed)
    X, Y, Z = _centres(origin - G * h0, h, 8 + 2 * G)
    U, _ = _blast(X, Y, Z, q)
    return U.contiguous(), origin, h


def _samples(case, seed):
    """Features and labels of a minibatch: about half of the cells in uniform surroundings (all zero), the others
    with relative differences of all sizes."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    n = case["n"]
    scale = 10.0 ** (-3.0 + 3.0 * torch.rand((n, 1), generator=gen, device=DEV))
    X = (torch.randn((n, 54), generator=gen, device=DEV) * scale).clamp(-1.0, 1.0)
    X = X * (torch.rand((n, 1), generator=gen, device=DEV) < 0.5)
    X[:, 13] = 0.0  # the cell itself
    X[:, 40] = 0.0
    y = ((X.abs().mean(1) + 0.02 * torch.rand(n, generator=gen, device=DEV)) > 0.03).to(torch.float32)
    return X.contiguous(), y


# ---------------------------------------------------------------------------
# prepare, run, work

def prepare(case, seed):
    kind = case["kind"]
    q = _params(seed)
    if kind == "uniform":
        origin, h = _mesh(case)
        U, g = _state(case["flow"], origin, h, case["N"], q)
        ctx = _context(case, _omega(case, q))
        if case["indicator"]:
            H.hydro_set_indicator(ctx, _indicator(seed), 0.5)
        nb = (case["nbx"], case["nby"], case["nbz"])
        run = UniformRun(ctx, U, origin.cpu().numpy(), h.cpu().numpy(), nb, _bc(case), g=g, cfl=0.4,
                         fused=case["fused"])
        return dict(kind=kind, ctx=ctx, run=run, N=case["N"])
    if kind == "amr":
        level, ijk = _amr_mesh(case, seed)
        o, h = W.amr_geometry(level, ijk)
        U, _ = _state("blast", torch.tensor(o, device=DEV), torch.tensor(h, device=DEV), 8, q)
        pad = torch.zeros((len(level), NF, 14, 14, 14), dtype=F64, device=DEV)
        pad[:, :, 3:-3, 3:-3, 3:-3] = U
        ctx = _context(case)
        return dict(kind=kind, ctx=ctx, run=A.AMRRun(ctx, pad, level, ijk), N=8)
    if kind == "batch":
        U, origin, h = _random_batch(case, seed)
        n, N = case["n"], case["N"]
        return dict(kind=kind, ctx=_context(case, q["spin"]), batch=H.make_batch(U, origin, h), static=case["static"],
                    dU=torch.empty((n, NF, N, N, N), dtype=F64, device=DEV),
                    am=torch.empty(n, dtype=F64, device=DEV),
                    faces=torch.empty((n, 6, NF + 3, N, N), dtype=F64, device=DEV) if case["faces"] else None)
    if kind == "labels":
        U, origin, h = _snapshot(case, seed)
        n = case["n"]
        ctx = H.Context(GAMMA, 0.0)
        H.hydro_set_mode(ctx, H.HYDRO_PREC_MIXED)
        return dict(kind=kind, ctx=ctx, batch=H.make_batch(U, origin, h), params=_indicator(seed),
                    X=torch.empty((n * 512, 54), dtype=torch.float32, device=DEV),
                    y=torch.empty(n * 512, dtype=torch.uint8, device=DEV),
                    out=torch.empty(n * 512, dtype=torch.float32, device=DEV))
    X, y = _samples(case, seed)
    params = _train_params(seed)
    return dict(kind=kind, X=X, y=y, params=params, m=torch.zeros_like(params), v=torch.zeros_like(params),
                grad=torch.empty_like(params), loss=torch.empty(1, dtype=torch.float32, device=DEV), t=0,
                work=torch.empty(H.hydro_mlp_work_bytes(case["n"]) // 4 + 1, dtype=torch.float32, device=DEV))


def _train_params(seed):
    rng = np.random.default_rng(seed + 5)
    parts = [rng.normal(0, math.sqrt(2.0 / 54), 32 * 54), rng.normal(0, 0.05, 32),
             rng.normal(0, math.sqrt(2.0 / 32), 32 * 32), rng.normal(0, 0.05, 32),
             rng.normal(0, math.sqrt(1.0 / 32), 32), np.zeros(1)]
    return torch.tensor(np.concatenate(parts), dtype=torch.float32, device=DEV)


def run(state):
    kind = state["kind"]
    if kind in ("uniform", "amr"):
        r, N = state["run"], state["N"]
        H.hydro_rk3_step(state["ctx"], r.desc, 0)
        return {"state": r.bufs[1][:, :, G:G + N, G:G + N, G:G + N], "dt": r.dt}
    if kind == "batch":
        if state["static"]:
            H.hydro_step_static(state["ctx"], state["batch"], 0.0, state["dU"], state["am"])
        else:
            H.hydro_step(state["ctx"], state["batch"], 0.0, state["dU"], state["am"], state["faces"])
        out = {"dU": state["dU"], "amax": state["am"]}
        if state["faces"] is not None:
            out["faces"] = state["faces"]
        return out
    if kind == "labels":
        H.hydro_gate_data(state["ctx"], state["batch"], state["X"], state["y"])
        H.hydro_mlp_forward(state["params"], state["X"], state["out"])
        return {"X": state["X"], "y": state["y"], "out": state["out"]}
    state["t"] += 1
    H.hydro_mlp_loss_grad(state["params"], state["X"], state["y"], state["grad"], state["loss"], 8.0, 1.0,
                          state["work"])
    H.hydro_mlp_adam(state["params"], state["m"], state["v"], state["grad"], state["t"], 3e-3)
    return {k: state[k] for k in ("grad", "loss", "params", "m", "v")}


def work(case):
    """Bytes and operations that a pass cannot do without.  Per 8^3 tile and stage: a PPM line of one field is about
    45 operations (10,112 lines of 10 fields with 9 points per face, 1,920 with one), a point flux about 130."""
    kind = case["kind"]
    if kind == "train":
        n = case["n"]
        return {"bytes": 4.0 * n * 55 + 4.0 * 2849 * 7, "flops": 6.0 * n * 2784}
    if kind == "labels":
        cells = 512.0 * case["n"]
        lines = 13 * 7 * 70.0 * cells
        return {"bytes": case["n"] * 14 ** 3 * 80.0 + cells * (54 * 4 + 1 + 54 * 4 + 4),
                "flops": lines + cells * (54 * 4 + 2 * 2784)}
    points = case.get("points", 9)
    tile = (10112 * 450.0 + 15552 * 130.0) if points == 9 else (1920 * 450.0 + 1728 * 130.0)
    if kind == "batch":
        n, N = case["n"], case["N"]
        t = n * (N // 8) ** 3
        return {"bytes": n * 80.0 * ((N + 6) ** 3 + N ** 3) + (n * 6 * 13 * N * N * 8.0 if case["faces"] else 0.0),
                "flops": t * tile}
    if kind == "uniform":
        t = case["nbx"] * case["nby"] * case["nbz"] * (case["N"] // 8) ** 3
        return {"bytes": t * 512 * (160.0 + (24.0 if case["flow"] == "star" else 0.0)), "flops": 3 * t * tile}
    t = len(_leaves(case["leaves"], case["lmin"], case["lmax"])[0])
    return {"bytes": t * 512 * 160.0, "flops": 3 * t * tile}


# ---------------------------------------------------------------------------
# the method in FP64

def _prims(U):
    """Primitives [n][F][...] of conserved states (dual-energy selection)."""
    rho = U[:, 0]
    q = U.clone()
    q[:, 1:4] = U[:, 1:4] / rho.unsqueeze(1)
    e = U[:, 4] - 0.5 * rho * (q[:, 1:4] ** 2).sum(1)
    q[:, 4] = torch.where(e > ETA1 * U[:, 4], e, U[:, 5].clamp_min(0.0) ** GAMMA)
    return q


def _slope(a, b):
    m = torch.minimum(2 * torch.minimum(a.abs(), b.abs()), 0.5 * (a + b).abs())
    return torch.where(a * b <= 0, torch.zeros_like(m), torch.copysign(m, b))


def _eta(s, rho, p):
    """Contact-steepening weight of one line's samples s (list of five)."""
    ok = GAMMA * 0.1 * (rho[1] - rho[0]).abs() * torch.minimum(p[0], p[1]) >= (p[1] - p[0]).abs() * torch.minimum(
        rho[0], rho[1])
    d2m, d2p = (s[0] + s[2]) - 2 * s[1], (s[2] + s[4]) - 2 * s[3]
    jump = s[3] - s[1]
    ok = ok & ~(d2m * d2p > 0) & ~(jump.abs() <= 0.01 * torch.minimum(s[3].abs(), s[1].abs()))
    et = -(d2p - d2m) / torch.where(ok, 6 * jump, torch.ones_like(jump))
    return torch.where(ok, (20 * (et - 0.05)).clamp(0.0, 1.0), torch.zeros_like(et))


def _ppm(s, eta=None):
    dl = [s[j + 1] - s[j] for j in range(4)]
    D = [_slope(dl[k], dl[k + 1]) for k in range(3)]
    q0 = s[2]
    qp = 0.5 * (q0 + s[3]) - (D[2] - D[1]) / 6
    qm = 0.5 * (s[1] + q0) - (D[1] - D[0]) / 6
    if eta is not None:
        st = eta > 0
        qp = torch.where(st, (1 - eta) * qp + eta * (s[3] - 0.5 * D[2]), qp)
        qm = torch.where(st, (1 - eta) * qm + eta * (s[1] + 0.5 * D[0]), qm)
    flat = (qp - q0) * (q0 - qm) <= 0
    dq = qp - qm
    lhs, rhs = dq * (q0 - 0.5 * (qp + qm)), dq * dq / 6
    nm = torch.where(lhs > rhs, 3 * q0 - 2 * qp, qm)
    np_ = torch.where(lhs < -rhs, 3 * q0 - 2 * qm, qp)
    return torch.where(flat, q0, np_), torch.where(flat, q0, nm)


def _stage(U, origin, h, N, omega, g=None, points=9, contact=False, spin=False, faces=False):
    """dU/dt, amax and (faces) the boundary-face sums of padded sub-grids."""
    n, M = U.shape[0], N + 2
    Q = _prims(U)
    hh = h.view(n, 1, 1, 1)

    def win(d, m):  # Q of the cells -1 .. N, shifted by m d
        a = [G - 1 + m * c for c in d]
        return Q[:, :, a[2]:a[2] + M, a[1]:a[1] + M, a[0]:a[0] + M]

    dirs = [(dx, dy, dz) for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)]
    R = {}
    q0 = win((0, 0, 0), 0)
    if spin:
        om = q0[:, 6:9] / (q0[:, :1] * (hh * hh / 6).unsqueeze(1))
        vc = torch.sqrt((om * om).sum(1)) * (0.5 * math.sqrt(3.0) * hh)
        cs = torch.sqrt((GAMMA * (GAMMA - 1) * q0[:, 4] / q0[:, 0]).clamp_min(0.0))
        om = om * torch.where(cs < vc, cs / vc.clamp_min(1e-300), torch.ones_like(cs)).unsqueeze(1)
    for d in dirs[14:]:
        if points == 1 and sum(map(abs, d)) != 1:
            continue
        if sum(map(abs, d)) == 0:
            continue
        s = [win(d, m) for m in range(-2, 3)]
        eta = None
        if contact:
            rho = (s[1][:, 0], s[3][:, 0])
            p = ((GAMMA - 1) * s[1][:, 4], (GAMMA - 1) * s[3][:, 4])
            eta = torch.zeros_like(q0)
            for k in (0, 9):
                eta[:, k] = _eta([x[:, k] for x in s], rho, p)
        qp, qm = _ppm(s, eta)
        if spin:
            r = [0.5 * c * hh for c in d]
            dv = torch.stack([om[:, 1] * r[2] - om[:, 2] * r[1], om[:, 2] * r[0] - om[:, 0] * r[2],
                              om[:, 0] * r[1] - om[:, 1] * r[0]], 1)
            qp[:, 1:4] += dv
            qm[:, 1:4] -= dv
        R[d], R[tuple(-c for c in d)] = qp, qm
    idx = torch.arange(-1, N + 1, dtype=F64, device=U.device) + 0.5
    cen = [origin[:, 0].view(n, 1, 1, 1) + hh * idx.view(1, 1, 1, M),
           origin[:, 1].view(n, 1, 1, 1) + hh * idx.view(1, 1, M, 1),
           origin[:, 2].view(n, 1, 1, 1) + hh * idx.view(1, M, 1, 1)]
    dU = torch.zeros((n, NF, N, N, N), dtype=F64, device=U.device)
    amax = torch.zeros(n, dtype=F64, device=U.device)
    ff = torch.zeros((n, 6, NF + 3, N, N), dtype=F64, device=U.device) if faces else None
    inv = 1.0 / h.view(n, 1, 1, 1, 1)
    for a in range(3):
        b, c = (1 if a == 0 else 0), (1 if a == 2 else 2)
        # slices of the (N+2)^3 cubes: left and right cells of the N + 1 faces along a
        sl = [slice(1, N + 1)] * 3
        sr = list(sl)
        sl[a], sr[a] = slice(0, N + 1), slice(1, N + 2)
        L, Rr = (slice(None), slice(None), sl[2], sl[1], sl[0]), (slice(None), slice(None), sr[2], sr[1], sr[0])
        Fs, TL, TR = 0, 0, 0
        for t1 in (-1, 0, 1):
            for t2 in (-1, 0, 1):
                if points == 1 and (t1 or t2):
                    continue
                d = [0, 0, 0]
                d[a], d[b], d[c] = 1, t1, t2
                dr = list(d)
                dr[a] = -1
                w = 1.0 if points == 1 else (4 if t1 == 0 else 1) * (4 if t2 == 0 else 1) / 36.0
                xq = [(cen[m].expand(n, M, M, M)[:, sl[2], sl[1], sl[0]] + 0.5 * d[m] * hh) for m in range(2)]
                sides = []
                for q in (R[tuple(d)][L], R[tuple(dr)][Rr]):
                    rho, v, eps = q[:, 0], q[:, 1:4], q[:, 4]
                    E = eps + 0.5 * rho * (v * v).sum(1)
                    p = (GAMMA - 1) * eps
                    cs = torch.sqrt(GAMMA * p / rho)
                    un = v[:, a] + (omega * xq[1] if a == 0 else -omega * xq[0] if a == 1 else 0.0)
                    Uc = q.clone()
                    Uc[:, 1:4] = rho.unsqueeze(1) * v
                    Uc[:, 4] = E
                    Fl = Uc * un.unsqueeze(1)
                    Fl[:, 1 + a] += p
                    Fl[:, 4] += p * v[:, a]
                    sides.append((Uc, Fl, un.abs() + cs))
                aq = torch.maximum(sides[0][2], sides[1][2])
                amax = torch.maximum(amax, aq.reshape(n, -1).amax(1))
                Fq = 0.5 * (sides[0][1] + sides[1][1]) - 0.5 * aq.unsqueeze(1) * (sides[1][0] - sides[0][0])
                Fs = Fs + w * Fq
                for e, who in ((d, 0), (dr, 1)):
                    r = [0.5 * x * hh for x in e]
                    T = torch.stack([r[1] * Fq[:, 3] - r[2] * Fq[:, 2], r[2] * Fq[:, 1] - r[0] * Fq[:, 3],
                                     r[0] * Fq[:, 2] - r[1] * Fq[:, 1]], 1)
                    if who == 0:
                        TL = TL + w * T
                    else:
                        TR = TR + w * T
        ax = 4 - a
        lo = [slice(None)] * 5
        hi = [slice(None)] * 5
        lo[ax], hi[ax] = slice(0, N), slice(1, N + 1)
        dU -= (Fs[tuple(hi)] - Fs[tuple(lo)]) * inv
        dU[:, 6:9] -= (TL[tuple(hi)] - TR[tuple(lo)]) * inv
        if faces:
            for side, at in ((0, 0), (1, N)):
                ff[:, 2 * a + side, :NF] = Fs.select(ax, at)
                ff[:, 2 * a + side, NF:] = (TL if side else TR).select(ax, at)
    Ui = U[:, :, G:G + N, G:G + N, G:G + N]
    s, z = Ui[:, 1:4], Ui[:, 6:9]
    xc, yc = cen[0][:, :, :, 1:N + 1], cen[1][:, :, 1:N + 1, :]
    wx, wy = omega * yc, -omega * xc
    dU[:, 1] += omega * s[:, 1]
    dU[:, 2] -= omega * s[:, 0]
    dU[:, 6] += omega * z[:, 1] + wy * s[:, 2]
    dU[:, 7] += -omega * z[:, 0] - wx * s[:, 2]
    dU[:, 8] += wx * s[:, 1] - wy * s[:, 0]
    if g is not None:
        dU[:, 1:4] += Ui[:, :1] * g
        dU[:, 4] += (s * g).sum(1)
    return dU, amax, ff


def _advance(U, U0, dU, dt, k):
    al, be = ((0.0, 1.0), (0.75, 0.25), (1 / 3, 2 / 3))[k]
    u = al * U0 + be * (U + dt * dU)
    e = u[:, 4] - 0.5 * (u[:, 1:4] ** 2).sum(1) / u[:, 0]
    u[:, 5] = torch.where(e > ETA2 * u[:, 4], e.clamp_min(0.0) ** (1.0 / GAMMA), u[:, 5])
    return u


def _windows(U, nb, N, bc):
    """A function of a range of sub-grids: their padded states from all interiors."""
    nx, ny, nz = nb

    def axis(n, k):  # global cells of the window of block k
        i = k * N + torch.arange(-G, N + G, device=DEV)
        return i % n if bc == "periodic" else i.clamp(0, n - 1)

    def of(a, b):
        out = torch.empty((b - a, NF, N + 2 * G, N + 2 * G, N + 2 * G), dtype=F64, device=DEV)
        for s in range(a, b):
            gx, gy, gz = axis(nx * N, s % nx), axis(ny * N, (s // nx) % ny), axis(nz * N, s // (nx * ny))
            o = ((gz // N).view(-1, 1, 1) * ny + (gy // N).view(1, -1, 1)) * nx + (gx // N).view(1, 1, -1)
            loc = ((gz % N).view(-1, 1, 1) * N + (gy % N).view(1, -1, 1)) * N + (gx % N).view(1, 1, -1)
            at = (o * (NF * N ** 3) + loc).unsqueeze(0) + (torch.arange(NF, device=DEV) * N ** 3).view(-1, 1, 1, 1)
            out[s - a] = U.view(-1)[at]
        return out

    return of


def _exact_uniform(case, seed):
    N = case["N"]
    n = case["nbx"] * case["nby"] * case["nbz"]
    if case["indicator"] or n * (N // 8) ** 3 > 8192:
        return None  # the indicator's decisions are discrete; a large mesh takes too long
    q = _params(seed)
    origin, h = _mesh(case)
    X, g = _state(case["flow"], origin, h, N, q)
    U, dt = X, None
    chunk = max(1, 256 // (N // 8) ** 3)
    for k in range(3):
        of = _windows(U.contiguous(), (case["nbx"], case["nby"], case["nbz"]), N, case["bc"])
        dU, am = torch.empty_like(X), []
        for a in range(0, n, chunk):
            b = min(n, a + chunk)
            d, m, _ = _stage(of(a, b), origin[a:b], h[a:b], N, _omega(case, q), None if g is None else g[a:b],
                             case["points"], case["contact"], case["spin"])
            dU[a:b] = d
            am.append(m)
        if k == 0:
            dt = 0.4 * (h / torch.cat(am)).amin()
        U = _advance(U, X, dU, dt, k)
    return {"state": U, "dt": dt.view(1)}


class _Octree:
    """Dense tables of a 2:1 balanced octree on [-1, 1]^3, and its ghost fill and flux correction."""

    def __init__(self, level, ijk):
        self.level, self.ijk = torch.tensor(level, device=DEV).long(), torch.tensor(ijk, device=DEV).long()
        self.table = {}
        for lv in range(int(level.min()) - 1, int(level.max()) + 2):
            t = np.full((2 ** max(lv, 0),) * 3, -2, dtype=np.int64)
            for s, (l, (i, j, k)) in enumerate(zip(level.tolist(), ijk.tolist())):
                if l == lv:
                    t[k, j, i] = s
                elif l > lv >= 0:
                    t[k >> (l - lv), j >> (l - lv), i >> (l - lv)] = -1
            self.table[lv] = torch.tensor(t, device=DEV)

    def owner(self, lv, g):
        return self.table[lv][g[..., 2] // 8, g[..., 1] // 8, g[..., 0] // 8]

    @staticmethod
    def cells(U, o, g):
        i = g % 8 + G
        return U[o, :, i[:, 2], i[:, 1], i[:, 0]]

    def fill(self, U):
        U = U.clone()
        i = torch.arange(14, device=DEV)
        pos = torch.stack(torch.meshgrid(i, i, i, indexing="ij"), -1).reshape(-1, 3)  # z, y, x
        pos = pos[((pos < G) | (pos >= G + 8)).any(1)]
        later = []
        for lv in sorted(set(self.level.tolist())):
            s = torch.nonzero(self.level == lv).view(-1)
            g = (self.ijk[s].unsqueeze(1) * 8 + (pos.flip(1) - G).unsqueeze(0)).clamp(0, 8 * 2 ** lv - 1).reshape(-1, 3)
            who = s.repeat_interleave(len(pos))
            p = pos.repeat(len(s), 1)
            o = self.owner(lv, g)
            m = o >= 0
            U[who[m], :, p[m, 0], p[m, 1], p[m, 2]] = self.cells(U, o[m], g[m])
            m = o == -1
            if m.any():
                acc = 0
                for c in range(8):
                    f = 2 * g[m] + torch.tensor([c & 1, (c >> 1) & 1, c >> 2], device=DEV)
                    acc = acc + self.cells(U, self.owner(lv + 1, f), f)
                U[who[m], :, p[m, 0], p[m, 1], p[m, 2]] = acc / 8
            m = o == -2
            if m.any():
                later.append((lv, who[m], p[m], g[m]))
        V = U.clone()
        for lv, who, p, g in later:
            gc = g // 2
            o = self.owner(lv - 1, gc)
            i = gc % 8 + G
            C = V[o, :, i[:, 2], i[:, 1], i[:, 0]]
            val = C.clone()
            for d in range(3):
                e = torch.zeros(3, dtype=torch.long, device=DEV)
                e[d] = 1
                up = V[o, :, i[:, 2] + e[2], i[:, 1] + e[1], i[:, 0] + e[0]] - C
                dn = C - V[o, :, i[:, 2] - e[2], i[:, 1] - e[1], i[:, 0] - e[0]]
                mm = torch.where(up * dn <= 0, torch.zeros_like(up), torch.where(up.abs() < dn.abs(), up, dn))
                val += mm * (0.5 * (g[:, d] % 2) - 0.25).unsqueeze(1)
            U[who, :, p[:, 0], p[:, 1], p[:, 2]] = val
        return U

    def correct(self, dU, ff, h):
        j = torch.arange(8, device=DEV)
        PC, PB = [x.reshape(-1) for x in torch.meshgrid(j, j, indexing="ij")]
        for a in range(3):
            b, c = (1 if a == 0 else 0), (1 if a == 2 else 2)
            for side in (0, 1):
                for lv in sorted(set(self.level.tolist())):
                    nbr = self.ijk.clone()
                    nbr[:, a] += 2 * side - 1
                    ok = (self.level == lv) & (nbr[:, a] >= 0) & (nbr[:, a] < 2 ** lv)
                    s = torch.nonzero(ok).view(-1)
                    s = s[self.owner(lv, nbr[s] * 8) == -1]
                    if not len(s):
                        continue
                    sg = 2.0 * side - 1.0
                    hc = h[s].view(-1, 1)
                    corr = torch.zeros((len(s), 64, NF + 3), dtype=F64, device=DEV)
                    for dc in (0, 1):
                        for db in (0, 1):
                            g = torch.zeros((len(s), 64, 3), dtype=torch.long, device=DEV)
                            g[..., a] = ((self.ijk[s, a] + 1) * 16 if side else self.ijk[s, a] * 16 - 1).view(-1, 1)
                            g[..., b] = 2 * (self.ijk[s, b].view(-1, 1) * 8 + PB) + db
                            g[..., c] = 2 * (self.ijk[s, c].view(-1, 1) * 8 + PC) + dc
                            v = ff[self.owner(lv + 1, g), 2 * a + 1 - side, :, g[..., c] % 8, g[..., b] % 8].clone()
                            r = [None] * 3
                            r[a], r[b], r[c] = 0.75 * sg * hc, (0.5 * db - 0.25) * hc, (0.5 * dc - 0.25) * hc
                            P = v[..., 1:4]
                            v[..., NF] += r[1] * P[..., 2] - r[2] * P[..., 1]
                            v[..., NF + 1] += r[2] * P[..., 0] - r[0] * P[..., 2]
                            v[..., NF + 2] += r[0] * P[..., 1] - r[1] * P[..., 0]
                            corr += v / 4
                    corr -= ff[s][:, 2 * a + side][:, :, PC, PB].permute(0, 2, 1)
                    corr *= -(sg / hc).unsqueeze(-1)
                    cell = [None] * 3
                    cell[a], cell[b], cell[c] = torch.full_like(PB, 7 * side), PB, PC
                    cur = dU[s][:, :, cell[2], cell[1], cell[0]]
                    add = corr[..., :NF].clone()
                    add[..., 6:9] += corr[..., NF:]
                    dU[s.view(-1, 1), :, cell[2], cell[1], cell[0]] = cur.permute(0, 2, 1) + add
        return dU


def _exact_amr(case, seed):
    level, ijk = _amr_mesh(case, seed)
    o, h = W.amr_geometry(level, ijk)
    o, h = torch.tensor(o, device=DEV), torch.tensor(h, device=DEV)
    X, _ = _state("blast", o, h, 8, _params(seed))
    tree = _Octree(level, ijk)
    n = len(level)
    U, dt = X, None
    for k in range(3):
        pad = torch.zeros((n, NF, 14, 14, 14), dtype=F64, device=DEV)
        pad[:, :, 3:-3, 3:-3, 3:-3] = U
        pad = tree.fill(pad)
        dU, am = torch.empty_like(X), torch.empty(n, dtype=F64, device=DEV)
        ff = torch.empty((n, 6, NF + 3, 8, 8), dtype=F64, device=DEV)
        for a in range(0, n, 256):
            sl = slice(a, min(n, a + 256))
            dU[sl], am[sl], ff[sl] = _stage(pad[sl], o[sl], h[sl], 8, 0.0, faces=True)
        dU = tree.correct(dU, ff, h)
        if k == 0:
            dt = 0.4 * (h / am).amin()
        U = _advance(U, X, dU, dt, k)
    return {"state": U, "dt": dt.view(1)}


def _split(theta):
    W1, b1, W2, b2, w3, b3 = torch.split(theta, [32 * 54, 32, 32 * 32, 32, 32, 1])
    return W1.view(32, 54), b1, W2.view(32, 32), b2, w3, b3


def _bf16(x):
    return x.to(torch.float32).to(torch.bfloat16).to(F64)


def exact(case, seed):
    kind = case["kind"]
    if kind == "uniform":
        return _exact_uniform(case, seed)
    if kind == "amr":
        return _exact_amr(case, seed)
    if kind == "batch":
        U, origin, h = _random_batch(case, seed)
        n, N = case["n"], case["N"]
        out = {"dU": [], "amax": [], "faces": []}
        for a in range(0, n, 256):
            sl = slice(a, min(n, a + 256))
            d, m, f = _stage(U[sl], origin[sl], h[sl], N, _params(seed)["spin"], None, 9, case["contact"],
                             case["spin"], True)
            out["dU"].append(d)
            out["amax"].append(m)
            out["faces"].append(f)
        out = {k: torch.cat(v) for k, v in out.items()}
        if not case["faces"]:
            del out["faces"]
        return out
    if kind == "labels":
        U, _, _ = _snapshot(case, seed)
        W1, b1, W2, b2, w3, b3 = _split(_bf16(_indicator(seed)))
        Xs, outs = [], []
        for a in range(0, case["n"], 64):
            Q = _prims(U[a:a + 64])
            f = []
            for v in (Q[:, 0], (GAMMA - 1) * Q[:, 4]):
                c = v[:, 3:11, 3:11, 3:11]
                for dz in (2, 3, 4):
                    for dy in (2, 3, 4):
                        for dx in (2, 3, 4):
                            k = v[:, dz:dz + 8, dy:dy + 8, dx:dx + 8]
                            f.append((k - c) / (k.abs() + c.abs()))
            X = torch.stack(f, -1).reshape(-1, 54)
            h1 = _bf16(torch.relu(_bf16(X) @ W1.T + b1))
            h2 = torch.relu(h1 @ W2.T + b2)
            Xs.append(X)
            outs.append(torch.sigmoid(h2 @ w3 + b3))
        return {"X": torch.cat(Xs), "y": None, "out": torch.cat(outs)}
    X, y = _samples(case, seed)
    X, y = X.to(F64), y.to(F64)
    p0 = _train_params(seed)
    theta = _bf16(p0).requires_grad_(True)
    W1, b1, W2, b2, w3, b3 = _split(theta)
    z3 = torch.relu(torch.relu(X @ W1.T + b1) @ W2.T + b2) @ w3 + b3
    sp = torch.nn.functional.softplus
    loss = (8.0 * y * sp(-z3) + (1 - y) * sp(z3)).mean()
    loss.backward()
    g = theta.grad
    m, v = 0.1 * g, 0.001 * g * g
    params = p0.to(F64) - 3e-3 * (m / 0.1) / (torch.sqrt(v / 0.001) + 1e-8)
    return {"grad": g, "loss": loss.detach().view(1), "params": params, "m": m, "v": v}
