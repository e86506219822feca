"""Performance cases: what users of the library have it do, each through a public entry point.

A pass of a simulation case is one output interval of a run: the state goes in
(`set_fields`), a number of explicit steps is taken and the state comes out, with
the composition integrals where the run prints them.  The adjoint case is one
gradient evaluation, the batched case one round of a parameter sweep.  Sizes and
materials are those of the workloads, the tests and the benchmark of this
repository; the initial states are seeded and have diffuse interfaces, the form
every run has after its first steps.

`exact` advances the same inputs in 64 bits with plain torch, written from the
equations: face fluxes of the anisotropic gradient energy, centre term, obstacle
or well potential, driving force, projection, mu update, and the options.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2404_01035_gb300 import ModelSpec, Simulation
from paper_2404_01035_gb300.autograd import GPSteps, theta_of
from paper_2404_01035_gb300.batch import Batch
from paper_2404_01035_gb300.sparse_gg import SparseGrainGrowth

PERIODIC, NOFLUX = 3, 1
EPS = 4.0                      # interface width of every workload
HALF = math.pi ** 2 / 8.0      # half width of the obstacle profile, in units of EPS


# ------------------------------------------------------------------ the cases
def listed():
    sim = dict(kind="sim", tune=False, option="", nz=1)
    return [
        # the bundled input deck's grid (two rotated solids and a liquid, ternary,
        # pulled gradient), FP32 as the deck driver's default: the smallest call
        dict(sim, name="deck_2d_f32", scene="deck", nx=56, ny=40, steps=40, dtype="f32"),
        # the 2-D dendrite workload in FP64: validation runs
        dict(sim, name="dendrite_2d_f64", scene="dendrite", nx=128, ny=128, steps=200, dtype="f64", delta=0.0),
        # a large ragged 2-D field of anisotropic dendrites, one launch per step
        dict(sim, name="dendrites_2d_f32", scene="dendrite", nx=1537, ny=1411, steps=60, dtype="f32", delta=0.04),
        # the benchmark's directional eutectic, tuned as long runs are
        dict(sim, name="eutectic_256_f32", scene="eutectic", nx=256, ny=256, nz=256, steps=100, dtype="f32",
             tune=True),
        # the same alloy on an odd grid with the anti-trapping current, in the
        # launch a deck gets without tuning
        dict(sim, name="eutectic_at_f32", scene="eutectic", nx=150, ny=133, nz=97, steps=50, dtype="f32",
             option="anti_trapping"),
        # the same in FP64: the form parity is checked in
        dict(sim, name="eutectic_f64", scene="eutectic", nx=67, ny=50, nz=61, steps=20, dtype="f64"),
        # the largest workload: 7 rotated grains in liquid, 512^3
        dict(sim, name="multigrain_512_f32", scene="multigrain", nx=512, ny=512, nz=512, steps=20, dtype="f32",
             tune=True),
        # dense grain growth: 8 grains filling the box
        dict(sim, name="grain_growth_f32", scene="grains", nx=192, ny=192, nz=192, steps=15, dtype="f32",
             tune=True),
        # equilibrium by FFT before every step: 7 grains with an eigenstrain in liquid
        dict(sim, name="elastic_f32", scene="multigrain", nx=128, ny=128, nz=128, steps=20, dtype="f32",
             option="elastic"),
        # sparse storage of the same physics (few grains per cell, triple term)
        dict(name="sparse_grains_f32", kind="sparse", nx=128, ny=128, nz=128, grains=8, steps=200, dtype="f32"),
        # a sweep: independent 2-D dendrites of uneven sizes in one launch
        dict(name="batch_f32", kind="batch", sims=32, lo=64, hi=512, multiple=32, layout=20240401, steps=400),
        # one gradient of a loss on the final microstructure (well potential)
        dict(name="adjoint_f32", kind="adjoint", n=256, ny=256, steps=200, every=100, dtype="f32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    scene = rng.choice(["deck", "dendrite", "eutectic", "eutectic", "multigrain", "grains", "elastic", "sparse",
                        "batch", "adjoint"])
    f64 = rng.random() < 0.25
    dtype = "f64" if f64 else "f32"
    sim = dict(kind="sim", scene=scene, tune=rng.random() < 0.4, option="", nz=1, dtype=dtype)
    if scene == "deck":
        return dict(sim, nx=_log_int(rng, 24, 400), ny=_log_int(rng, 24, 400), steps=rng.randint(20, 60), tune=False)
    if scene == "dendrite":
        top = 300 if f64 else 2400
        return dict(sim, nx=_log_int(rng, 33, top), ny=_log_int(rng, 33, top), steps=rng.randint(20, 100),
                    delta=rng.choice([0.0, 0.02, 0.05]), tune=False)
    if scene == "eutectic":
        lo, hi = (24, 80) if f64 else (40, 256)
        return dict(sim, nx=_log_int(rng, lo, hi), ny=_log_int(rng, lo, hi), nz=_log_int(rng, max(lo, 40), hi),
                    steps=rng.randint(10, 20 if f64 else 60),
                    option=rng.choice(["", "anti_trapping", "noise"]), tune=not f64 and rng.random() < 0.4)
    if scene == "multigrain":
        lo, hi = (32, 56) if f64 else (64, 384)
        return dict(sim, nx=_log_int(rng, lo, hi), ny=_log_int(rng, lo, hi), nz=_log_int(rng, lo, hi),
                    steps=rng.randint(5, 20))
    if scene == "grains":
        lo, hi = (24, 40) if f64 else (48, 192)
        return dict(sim, nx=_log_int(rng, lo, hi), ny=_log_int(rng, lo, hi), nz=_log_int(rng, lo, hi),
                    steps=rng.randint(5, 12))
    if scene == "elastic":
        lo, hi = (32, 48) if f64 else (48, 144)
        return dict(sim, scene="multigrain", option="elastic", tune=False, nx=_log_int(rng, lo, hi),
                    ny=_log_int(rng, lo, hi), nz=_log_int(rng, lo, hi), steps=rng.randint(5, 15))
    if scene == "sparse":
        c = dict(kind="sparse", steps=rng.randint(20, 100), dtype=dtype)
        if rng.random() < 0.3:   # 2-D: many grains
            lo, hi = (64, 128) if f64 else (128, 400)
            return dict(c, nx=_log_int(rng, lo, hi), ny=_log_int(rng, lo, hi), nz=1, grains=rng.randint(8, 32))
        lo, hi = (24, 48) if f64 else (48, 128)
        return dict(c, nx=_log_int(rng, lo, hi), ny=_log_int(rng, lo, hi), nz=_log_int(rng, lo, hi),
                    grains=rng.randint(4, 8))
    if scene == "batch":
        return dict(kind="batch", sims=rng.randint(2, 32), lo=64, hi=rng.choice([128, 256, 512]),
                    multiple=rng.choice([32, 45, 77]), layout=rng.randint(1, 1 << 30), steps=rng.randint(50, 300))
    top = 112 if f64 else 320
    return dict(kind="adjoint", n=_log_int(rng, 40, top), ny=_log_int(rng, 40, top), steps=rng.randint(20, 80),
                every=rng.choice([20, 50]), dtype=dtype)


def work(case):
    """Every field read and written once a step (a reverse step also reads the
    state), the inputs and outputs once; operations: those of a cell whose whole
    neighbourhood is one pure phase, which no cell can do without."""
    s = 8 if case.get("dtype") == "f64" else 4
    if case["kind"] == "batch":
        cells, nf, nm, dim = sum(a * b for a, b in _batch_layout(case)), 3, 1, 2
    elif case["kind"] == "adjoint":
        cells, nf, nm, dim = case["n"] * case["ny"], 3, 1, 2
    elif case["kind"] == "sparse":
        # what a cell stores of its grains: at least one value and its index
        cells = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": cells * (2 * (s + 1) * case["steps"] + 2 * s * case["grains"]), "flops": cells * case["steps"]}
    else:
        cells = case["nx"] * case["ny"] * case["nz"]
        nf, nm = {"deck": (5, 2), "dendrite": (3, 1), "eutectic": (5, 2)}.get(case["scene"], (9, 1))
        dim = 2 if case["nz"] == 1 else 3
    passes = case["steps"] * (5 if case["kind"] == "adjoint" else 2) + 2
    return {"bytes": passes * s * nf * cells, "flops": case["steps"] * cells * nm * (2 * dim + 2 + 2 * nm)}


# ------------------------------------------------------------------ materials
def _spec(dim, shape, N, NM, bc, **kw):
    nz, ny, nx = shape
    D = np.zeros((N, NM, NM))
    D[N - 1] = np.eye(NM)
    base = dict(dim=dim, nx=nx, ny=ny, nz=nz, n_phases=N, n_components=NM + 1, bc=list(bc), dx=1.0, dt=0.0, eps=EPS,
                tau=1.0, potential="obstacle", gamma=np.ones((N, N)) - np.eye(N), delta=np.zeros((N, N)),
                rot=np.tile(np.eye(3), (N, N, 1, 1)), gamma3=None, D=D, A=np.stack([np.eye(NM)] * N),
                ceq=np.zeros((N, NM)), slopes=np.zeros((N, NM)), f0=np.zeros(N))
    base.update(kw)
    # 0.2 of the explicit stability bound for unit gamma and liquid diffusivity
    base["dt"] = base["dt"] or 0.2 / (2.0 * dim * (1.0 + 15.0 * float(np.max(base["delta"]))))
    return ModelSpec(**base)


def _rotation(g, dim):
    if dim == 2:
        c, s = math.cos(2 * math.pi * g[0]), math.sin(2 * math.pi * g[0])
        return np.array([[c, -s, 0.0], [s, c, 0.0], [0.0, 0.0, 1.0]])
    a, b = math.sqrt(1.0 - g[0]), math.sqrt(g[0])   # a uniform quaternion
    x, y, z, w = (a * math.sin(2 * math.pi * g[1]), a * math.cos(2 * math.pi * g[1]), b * math.sin(2 * math.pi * g[2]),
                  b * math.cos(2 * math.pi * g[2]))
    return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
                     [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
                     [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]])


def _binary(shape, dim, delta, Delta, potential="obstacle", dt=0.0):
    d = np.array([[0.0, delta], [delta, 0.0]])
    return _spec(dim, shape, 2, 1, [PERIODIC] * 3, delta=d, ceq=np.array([[0.926], [0.817]]), potential=potential,
                 f0=np.array([-Delta, 0.0]), dt=dt)


def _problem(case, rng):
    """The problem of a simulation case; rng: numpy, seeded by the inputs' seed."""
    nz, ny, nx = shape = (case["nz"], case["ny"], case["nx"])
    scene = case["scene"]
    if scene == "dendrite":
        return _binary(shape, 2, case["delta"], 0.2)
    if scene == "deck":
        d = np.zeros((3, 3))
        rot = np.tile(np.eye(3), (3, 3, 1, 1))
        for (a, b), v in {(0, 1): 0.02, (0, 2): 0.03, (1, 2): 0.01}.items():
            d[a, b] = d[b, a] = v
            if b == 2:
                rot[a, b] = rot[b, a] = _rotation(rng.random(3), 2)
        gam = np.array([[0, 1.0, 0.9], [1.0, 0, 1.1], [0.9, 1.1, 0]])
        D = np.stack([np.diag(v) for v in ((0.02, 0.01), (0.01, 0.02), (0.5, 0.4))])
        A = np.array([[[1.0, 0.05], [0.0, 0.9]], [[0.8, 0.0], [0.0, 1.1]], [[1.0, 0.0], [0.0, 1.0]]])
        sl = np.array([[-0.05, 0.0], [0.0, -0.05], [0.0, 0.0]])
        return _spec(2, shape, 3, 2, [PERIODIC, NOFLUX, PERIODIC], gamma=gam, delta=d, rot=rot, D=D, A=A, slopes=sl,
                     ceq=np.array([[0.7, 0.1], [0.15, 0.7], [0.4, 0.35]]), T_ref=1.0, T0=0.98, G=1e-3, z0=10.0, V=0.05,
                     dt=0.02)
    if scene == "eutectic":
        d = np.zeros((3, 3))
        d[:2, 2] = d[2, :2] = 0.02
        sl = np.zeros((3, 2))
        sl[2] = -0.05
        kw = {"anti_trapping": {"anti_trapping": 1}, "noise": {"noise_amp": 0.01, "noise_seed": 20240401}}
        return _spec(3, shape, 3, 2, [PERIODIC, PERIODIC, NOFLUX], delta=d, slopes=sl,
                     ceq=np.array([[0.75, 0.125], [0.125, 0.75], [0.4, 0.4]]), G=1e-3, z0=24.0, V=0.05,
                     **kw.get(case["option"], {}))
    if scene == "multigrain":
        d = np.zeros((8, 8))
        d[:7, 7] = d[7, :7] = 0.02
        rot = np.tile(np.eye(3), (8, 8, 1, 1))
        for a in range(7):
            rot[a, 7] = rot[7, a] = _rotation(rng.random(3), 3)
        kw = {}
        if case["option"] == "elastic":
            C = np.zeros((6, 6))
            C[:3, :3] = 0.6
            C[range(3), range(3)] = 1.0
            C[range(3, 6), range(3, 6)] = 0.4
            eig = np.zeros((8, 3, 3))
            eig[:7] = 0.01 * np.eye(3)
            kw = dict(elastic_C=C, eigenstrain=eig)
        return _spec(3, shape, 8, 1, [PERIODIC] * 3, delta=d, rot=rot, ceq=np.array([[0.926]] * 7 + [[0.817]]),
                     f0=np.array([-0.2] * 7 + [0.0]), **kw)
    return _grain_problem(shape, 8)


def _grain_problem(shape, N, **kw):
    return _spec(2 if shape[0] == 1 else 3, shape, N, 1, [PERIODIC] * 3, D=np.zeros((N, 1, 1)), ceq=np.full((N, 1), 0.5), grain_growth=1, **kw)


# ------------------------------------------------------------- initial states
def _profile(u):
    """Equilibrium profile of the obstacle potential, u = signed distance / EPS."""
    return 0.5 * (1.0 + torch.sin(4.0 / math.pi * u.clamp(-HALF, HALF)))


def _rest(phi):
    """1 - sum of the given phases, without the remainders of rounding."""
    v = 1.0 - phi.sum(0)
    return torch.where(v > 1e-12, v, torch.zeros_like(v))


def _axes(shape):
    nz, ny, nx = shape
    c = [torch.arange(n, device="cuda", dtype=torch.float64) + 0.5 for n in (nz, ny, nx)]
    return c[0][:, None, None], c[1][None, :, None], c[2][None, None, :]


def _gap(a, c, n):
    d = (a - c).abs()
    return torch.minimum(d, n - d)


def _ball(shape, c, R, dim):
    z, y, x = _axes(shape)
    r2 = _gap(x, c[0], shape[2]) ** 2 + _gap(y, c[1], shape[1]) ** 2
    if dim == 3:
        r2 = r2 + _gap(z, c[2], shape[0]) ** 2
    return R - torch.sqrt(r2)


def _waves(shape, rng, amp):
    z, y, x = _axes(shape)
    nz, ny, nx = shape
    p = 2 * math.pi * rng.random(3)
    w = torch.sin(2 * math.pi * x / nx + p[0]) + (torch.sin(4 * math.pi * y / ny + p[1]) *
                                                  torch.cos(2 * math.pi * z / nz + p[2]))
    return amp * w


def _fields(case, spec, rng):
    """phi [N, z, y, x] and mu [K-1, z, y, x] in 64 bits on the GPU."""
    shape = (spec.nz, spec.ny, spec.nx)
    N, ext = spec.n_phases, np.array([spec.nx, spec.ny, spec.nz], dtype=float)
    phi = torch.zeros((N,) + shape, device="cuda", dtype=torch.float64)
    scene = case["scene"]
    if scene == "dendrite":
        u = torch.full(shape, -1e9, device="cuda", dtype=torch.float64)
        seeds = max(1, int(spec.nx * spec.ny / 256 ** 2))
        for _ in range(seeds):
            c = ext / 2 + rng.uniform(-2, 2, 3) if seeds == 1 else rng.random(3) * ext
            R = rng.uniform(8, 12) if seeds == 1 else rng.uniform(8, 28)
            u = torch.maximum(u, _ball(shape, c, R, 2))
        phi[0] = _profile(u / EPS)
        phi[1] = 1.0 - phi[0]
        mu = [1.634 + _waves(shape, rng, 0.005)]
    elif scene == "deck":
        for a in (0, 1):
            u = torch.full(shape, -1e9, device="cuda", dtype=torch.float64)
            for _ in range(max(1, int(spec.nx * spec.ny / 64 ** 2))):
                u = torch.maximum(u, _ball(shape, rng.random(3) * ext, rng.uniform(5, 9), 2))
            phi[a] = _profile(u / EPS)
        both = (phi[0] + phi[1]).clamp(min=1.0)
        phi[:2] /= both
        phi[2] = _rest(phi[:2])
        # the liquid at its fill composition
        mu = [2.0 * 0.38 + _waves(shape, rng, 0.005), 2.0 * 0.33 + _waves(shape, rng, 0.005)]
    elif scene == "eutectic":
        # alternating lamellae 8 to 24 cells wide under a gently waved front
        z, y, x = _axes(shape)
        cuts, at = [], 0.0
        while at < spec.nx:
            cuts.append(at)
            at += float(rng.integers(8, 25))
        cuts = cuts[: len(cuts) // 2 * 2] or [0.0, spec.nx / 2.0]
        xs = x.reshape(-1)
        edge = torch.tensor(cuts, device="cuda", dtype=torch.float64)
        near = _gap(xs[:, None], edge[None, :], spec.nx).min(1).values
        side = torch.searchsorted(edge, xs, right=True) % 2
        alpha = _profile(torch.where(side == 1, near, -near) / EPS)
        front = 20.0 + _waves((1, spec.ny, spec.nx), rng, 2.0)
        liquid = _profile((z - front) / EPS)
        phi[2] = liquid
        phi[0] = (1.0 - liquid) * alpha
        phi[1] = (1.0 - liquid) * (1.0 - alpha)
        layer = torch.exp(-(z - front).clamp(min=0.0) / 12.0) * (alpha - 0.5)
        mu = [0.8 + 0.02 * layer, 0.8 - 0.02 * layer]
    elif scene == "multigrain":
        for a in range(7):
            c, R = rng.random(3) * ext, rng.uniform(8.0, 16.0)
            h = int(R + HALF * EPS) + 2
            if min(shape) > 2 * h + 1:   # only the box that the grain reaches
                ix = [torch.arange(int(c[d]) - h, int(c[d]) + h + 1, device="cuda") % int(ext[d]) for d in range(3)]
                g = [_gap(ix[d].double() + 0.5, c[d], ext[d]) ** 2 for d in range(3)]
                r = torch.sqrt(g[2][:, None, None] + g[1][None, :, None] + g[0][None, None, :])
                phi[a, ix[2][:, None, None], ix[1][None, :, None], ix[0][None, None, :]] = _profile((R - r) / EPS)
            else:
                phi[a] = _profile(_ball(shape, c, R, 3) / EPS)
        total = phi[:7].sum(0).clamp(min=1.0)
        for a in range(7):
            phi[a] /= total
        phi[7] = _rest(phi[:7])
        mu = [1.634 + _waves(shape, rng, 0.005)]
    else:
        phi = _voronoi(shape, N, rng)
        mu = [torch.full(shape, 0.25, device="cuda", dtype=torch.float64)]
    return phi, torch.stack([m.expand(shape) for m in mu])


def _voronoi(shape, N, rng):
    """Periodic Voronoi grains; each cell shares the profile in the signed
    distance to the plane between its nearest two centres."""
    z, y, x = _axes(shape)
    ext = torch.tensor([shape[2], shape[1], shape[0]], device="cuda", dtype=torch.float64)
    # centres at least half the mean grain size apart (periodic), as nuclei that have grown are
    size, put, dim = np.array(shape[::-1], dtype=float), [], 2 if shape[0] == 1 else 3
    while len(put) < N:
        c = rng.random(3) * size
        c[2] = 0.5 if shape[0] == 1 else c[2]
        gaps = [np.minimum(np.abs(c - o), size - np.abs(c - o)) for o in put]
        if all(np.linalg.norm(g) >= 0.5 * (np.prod(size) / N) ** (1 / dim) for g in gaps):
            put.append(c)
    cen = torch.tensor(np.stack(put), device="cuda", dtype=torch.float64)
    d2 = torch.stack([_gap(x, cen[a, 0], ext[0]) ** 2 + _gap(y, cen[a, 1], ext[1]) ** 2 + _gap(z, cen[a, 2], ext[2]) ** 2
                      for a in range(N)])
    v, k = torch.topk(d2, 2, dim=0, largest=False)
    del d2
    dc = cen[k[1]] - cen[k[0]]
    dc = dc - ext * torch.round(dc / ext)
    f = _profile((v[1] - v[0]) / (2.0 * dc.norm(dim=-1)) / EPS)
    phi = torch.zeros((N,) + tuple(shape), device="cuda", dtype=torch.float64)
    phi.scatter_(0, k[:1], f[None])
    phi.scatter_(0, k[1:], (1.0 - f)[None])
    return phi


def _batch_layout(case):
    """Edges (ny, nx) of the sweep's simulations."""
    r = np.random.default_rng(case["layout"])
    edges = np.arange(case["lo"], case["hi"] + 1, case["multiple"])
    return [(int(e), int(e)) for e in r.choice(edges, case["sims"])]


def _batch_inputs(case, seed):
    r, out = np.random.default_rng(seed), []
    for ny, nx in _batch_layout(case):
        spec = _binary((1, ny, nx), 2, 0.01 + 0.04 * r.random(), 0.1 + 0.3 * r.random())
        c = np.array([nx, ny, 0]) / 2 + r.uniform(-2, 2, 3)
        phi = _profile(_ball((1, ny, nx), c, 6.0, 2) / EPS)
        out.append((spec, torch.stack([phi, 1.0 - phi]), torch.full((1, 1, ny, nx), 1.634, device="cuda", dtype=torch.float64)))
    return out


def _adjoint_inputs(case, seed):
    r = np.random.default_rng(seed)
    shape = (1, case["ny"], case["n"])
    # delta and mobility of the evaluation point, dt of the target's
    spec = _binary(shape, 2, 0.02, 0.2, potential="well", dt=0.2 / (4.0 * 1.45))
    spec.tau = 1.0 / 0.8
    c = np.array([shape[2], shape[1], 0]) / 2 + r.uniform(-3, 3, 3)
    u = [_ball(shape, c, R, 2) / EPS for R in (10.0, 10.0 + 2.0 * r.random())]
    phi, target = (torch.stack([0.5 * (1 + torch.tanh(1.5 * v)), 0.5 * (1 - torch.tanh(1.5 * v))]) for v in u)
    mu = (1.634 + _waves(shape, r, 0.005)).expand(shape)[None]
    return spec, phi, mu, target


def _types(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def _sim_inputs(case, seed):
    rng = np.random.default_rng(seed)
    spec = _problem(case, rng)
    phi, mu = _fields(case, spec, rng)
    return spec, phi.to(_types(case)).contiguous(), mu.to(_types(case)).contiguous()


def _sparse_inputs(case, seed):
    rng = np.random.default_rng(seed)
    N, shape = case["grains"], (case["nz"], case["ny"], case["nx"])
    g3 = np.full((N, N, N), 15.0)   # uniform triple term over distinct triples
    for k in range(N):
        g3[k, k, :] = g3[k, :, k] = g3[:, k, k] = 0.0
    return _grain_problem(shape, N, gamma3=g3), _voronoi(shape, N, rng).to(_types(case)).contiguous()


# ------------------------------------------------------------ prepare and run
def prepare(case, seed):
    kind = case["kind"]
    if kind == "sim":
        spec, phi, mu = _sim_inputs(case, seed)
        sim = Simulation(spec, dtype=case["dtype"])
        if case["tune"]:   # once per simulation, as before a long run
            sim.set_fields(phi, mu)
            sim.tune(None, steps_per_trial=5)
        return {"case": case, "sim": sim, "phi": phi, "mu": mu, "out": (torch.empty_like(phi), torch.empty_like(mu))}
    if kind == "sparse":
        spec, phi = _sparse_inputs(case, seed)
        return {"case": case, "sim": SparseGrainGrowth(spec, dtype=case["dtype"]), "phi": phi}
    if kind == "batch":
        inputs = _batch_inputs(case, seed)
        host = [(phi.float().cpu().numpy(), mu.float().cpu().numpy()) for _, phi, mu in inputs]
        return {"case": case, "batch": Batch([spec for spec, _, _ in inputs]), "host": host}
    spec, phi, mu, target = _adjoint_inputs(case, seed)
    t = _types(case)
    return {"case": case, "sim": Simulation(spec, dtype=case["dtype"]), "target": target.to(t),
            "in": (phi.to(t).requires_grad_(), mu.to(t).requires_grad_(),
                   torch.tensor(theta_of(spec), dtype=t).requires_grad_())}


def run(state):
    case = state["case"]
    steps = case["steps"]
    if case["kind"] == "sim":
        sim = state["sim"]
        phi, mu = state["out"]
        sim.set_fields(state["phi"], state["mu"])
        sim.step(steps)
        mass = []
        if case["scene"] in ("deck", "eutectic"):   # these runs print the composition integrals
            mass = [float(v) for v in sim.diag()["mass"]]
        sim.get_fields_into(phi, mu, on_device=True)
        return {"phi": phi, "mu": mu, "mass": mass}
    if case["kind"] == "sparse":
        sim = state["sim"]
        sim.set_fields(state["phi"])
        sim.step(steps)
        return {"phi": sim.get_fields()}
    if case["kind"] == "batch":
        b = state["batch"]
        for i, (phi, mu) in enumerate(state["host"]):
            b.set_fields(i, phi, mu)
        b.step(steps)
        out = [b.get_fields(i) for i in range(case["sims"])]
        return {"phi": [f[0] for f in out], "mu": [f[1] for f in out]}
    phi0, mu0, theta = state["in"]
    phi, mu = GPSteps.apply(phi0, mu0, theta, state["sim"], steps, case["every"])
    loss = ((phi - state["target"]) ** 2).sum()
    dphi, dmu, dtheta = torch.autograd.grad(loss, (phi0, mu0, theta))
    return {"phi": phi.detach(), "mu": mu.detach(), "dphi": dphi, "dmu": dmu, "dtheta": dtheta}


# ------------------------------------------------------------- exact, 64 bits
def _shift(a, axis, s, bc):
    """The neighbours at +s along an axis (negative index), ghosts by the boundary code."""
    if bc == PERIODIC:
        return torch.roll(a, -s, axis)
    n = a.shape[axis]
    if s > 0:
        return torch.cat([a.narrow(axis, 1, n - 1), a.narrow(axis, n - 1, 1)], axis)
    return torch.cat([a.narrow(axis, 0, 1), a.narrow(axis, 0, n - 1)], axis)


def _padded(a, axis, bc):
    n = a.shape[axis]
    lo, hi = (n - 1, 0) if bc == PERIODIC else (0, n - 1)
    return torch.cat([a.narrow(axis, lo, 1), a, a.narrow(axis, hi, 1)], axis)


class _Exact:
    """The step in 64 bits for fields [N, B, z, y, x] (B simulations of one size)."""

    def __init__(self, spec, delta=None, tau=None, D=None, f0=None, dt=None, active=False, gamma3=0.0):
        self.s, self.dim, self.N, self.NM = spec, spec.dim, spec.n_phases, spec.n_mu
        dev = dict(device="cuda", dtype=torch.float64)
        N, NM, L = self.N, self.NM, self.N - 1
        self.delta = delta if delta is not None else spec.delta
        self.mob = 1.0 / (tau if tau is not None else spec.tau)
        self.dt = dt if dt is not None else spec.dt
        self.active, self.g3 = active, gamma3
        H = np.stack([np.array([[(2.0 if i == j else 1.0) * spec.A[a][min(i, j), max(i, j)] for j in range(NM)]
                                for i in range(NM)]) for a in range(N)])
        chi = np.linalg.inv(H)
        self.chi = torch.tensor(chi, **dev)
        self.D = D if D is not None else torch.tensor(spec.D, **dev)
        ce, sl = spec.ceq, spec.slopes
        B0 = np.stack([H[L] @ ce[L] - H[a] @ ce[a] if a != L else 0 * ce[L] for a in range(N)])
        B1 = np.stack([H[L] @ sl[L] - H[a] @ sl[a] if a != L else 0 * sl[L] for a in range(N)])
        self.B0, self.B1 = torch.tensor(B0, **dev), torch.tensor(B1, **dev)
        q = lambda u, v: np.array([0.5 * (u[a] @ H[a] @ v[a] - u[L] @ H[L] @ v[L]) if a != L else 0.0 for a in range(N)])  # noqa: E731
        self.f0 = f0 if f0 is not None else [float(v) for v in spec.f0]
        self.C = [q(ce, ce), 2.0 * q(sl, ce), q(sl, sl)]
        self.dcT = torch.tensor(np.einsum("aij,aj->ai", chi, B1) * spec.G * spec.V * spec.dt, **dev)
        last = spec.nz if self.dim == 3 else spec.ny
        k = torch.arange(last, **dev) + 0.5
        self.pos = k[:, None, None] if self.dim == 3 else k[None, :, None]
        self.iso = all(not torch.is_tensor(v) and v == 0 for row in self.delta for v in row)

    def axes(self):
        return [(-1, self.s.bc[0]), (-2, self.s.bc[1]), (-3, self.s.bc[2])][: self.dim]

    def temperature(self, t, pos):
        s = self.s
        return s.T0 - s.T_ref + s.G * (pos * s.dx - s.z0 - s.V * t)

    def pair(self, a, b):
        """gamma, delta (None where isotropic) and rotation (None where it is the identity)."""
        R = self.s.rot[a, b]
        d = self.delta[a][b]
        plain = not torch.is_tensor(d) and d == 0
        return float(self.s.gamma[a, b]), None if plain else d, None if np.array_equal(R, np.eye(3)) else R

    def gradient(self, q, a, b, only=None):
        """g = dA/dq of the pair, A = gamma a_c(Rq)^2 |q|^2 (component `only`, or all)."""
        gam, d, R = self.pair(a, b)
        if d is None:
            return 2 * gam * q[only] if only is not None else [2 * gam * v for v in q]
        n = len(q)
        Q = sum(v * v for v in q)
        small = Q < 1e-12
        Qs = torch.where(small, torch.ones_like(Q), Q)
        r = q if R is None else [sum(R[i, j] * q[j] for j in range(n)) for i in range(n)]
        s4 = sum(v ** 4 for v in r) / Qs ** 2
        ac = 1 - d * (3 - 4 * s4)
        g = [2 * gam * ac * v * (ac + 16 * d * (v * v / Qs - s4)) for v in r]
        if R is not None:
            g = [sum(R[i, j] * g[i] for i in range(n)) for j in range(n)]
        g = [torch.where(small, torch.zeros_like(v), v) for v in (g if only is None else [g[only]])]
        return g[0] if only is not None else g

    def h(self, P):
        e1 = P.sum(0)
        e2 = 0.5 * (e1 * e1 - (P * P).sum(0))
        return P * P * (3 - 2 * P) + 2 * P * (e2 - P * (e1 - P))

    def div_flux(self, P):
        dx, N = self.s.dx, self.N
        out = 0.0
        for D, (ax, bc) in enumerate(self.axes()):
            pad = _padded(P, ax, bc)
            n = P.shape[ax]
            lo, hi = pad.narrow(ax, 0, n + 1), pad.narrow(ax, 1, n + 1)
            pf, gn = 0.5 * (lo + hi), (hi - lo) / dx
            if self.iso and float(np.ptp(self.s.gamma[~np.eye(N, dtype=bool)])) == 0.0:
                # one gamma: sum_b phi_b (phi_a grad phi_b - phi_b grad phi_a)
                J = -2 * float(self.s.gamma[0, 1]) * (pf * (pf * gn).sum(0) - gn * (pf * pf).sum(0))
            else:
                both = lo + hi
                gr = [gn if e == D else (_shift(both, a2, 1, b2) - _shift(both, a2, -1, b2)) / (4 * dx)
                      for e, (a2, b2) in enumerate(self.axes())]
                Js = [0.0] * N
                for a in range(N):
                    for b in range(a + 1, N):
                        if self.pair(a, b)[1] is None:
                            g = 2 * self.pair(a, b)[0] * (pf[a] * gn[b] - pf[b] * gn[a])
                        else:
                            g = self.gradient([pf[a] * v[b] - pf[b] * v[a] for v in gr], a, b, D)
                        Js[a] = Js[a] - pf[b] * g
                        Js[b] = Js[b] + pf[a] * g
                J = torch.stack(Js)
            out = out + (J.narrow(ax, 1, n) - J.narrow(ax, 0, n)) / dx
        return out

    def centre(self, P):
        N = self.N
        gc = [(_shift(P, ax, 1, bc) - _shift(P, ax, -1, bc)) / (2 * self.s.dx) for ax, bc in self.axes()]
        if self.iso and float(np.ptp(self.s.gamma[~np.eye(N, dtype=bool)])) == 0.0:
            G = 0.0
            for g in gc:
                G = G + 2 * float(self.s.gamma[0, 1]) * (P * (g * g).sum(0) - g * (P * g).sum(0))
            return G
        G = [0.0] * N
        for a in range(N):
            for b in range(a + 1, N):
                g = self.gradient([P[a] * v[b] - P[b] * v[a] for v in gc], a, b)
                G[a] = G[a] + sum(u * v[b] for u, v in zip(g, gc))
                G[b] = G[b] - sum(u * v[a] for u, v in zip(g, gc))
        return torch.stack(G)

    def project(self, P, v):
        if self.s.potential != "obstacle":
            return v - (v.sum(0) - 1) / self.N
        if self.active:   # over the grains at the cell or at a face neighbour
            on = P > 0
            near = on
            for ax, bc in self.axes():
                near = near | _shift(on, ax, 1, bc) | _shift(on, ax, -1, bc)
            v = torch.where(near, v, torch.full_like(v, -1e30))
        u = torch.sort(v, 0, descending=True).values
        j = torch.arange(1, self.N + 1, device=v.device, dtype=v.dtype).reshape((-1,) + (1,) * (v.dim() - 1))
        t = (torch.cumsum(u, 0) - 1) / j
        k = ((u - t) > 0).sum(0, keepdim=True) - 1
        return (v - torch.gather(t, 0, k)).clamp(min=0.0)

    def elastic(self, P):
        """-sigma : eigenstrain of each phase at mechanical equilibrium (periodic, no mean strain)."""
        s, dim = self.s, self.dim
        v = [[0, 5, 4], [5, 1, 3], [4, 3, 2]]
        C = torch.tensor([[[[s.elastic_C[v[i][j]][v[k][m]] for m in range(dim)] for k in range(dim)] for j in range(dim)]
                          for i in range(dim)], device="cuda", dtype=torch.float64)
        e0 = torch.tensor(s.eigenstrain[:, :dim, :dim], device="cuda", dtype=torch.float64)
        E = torch.einsum("abzyx,aij->ijbzyx", self.h(P), e0)
        ext = [s.nx, s.ny, s.nz][:dim]
        ks = []
        for d, n in enumerate(ext):
            k = 2 * math.pi * torch.fft.fftfreq(n, s.dx, device="cuda", dtype=torch.float64)
            if n % 2 == 0:
                k[n // 2] = 0.0
            ks.append(k.reshape([-1 if ax == 2 - d else 1 for ax in range(3)]).expand(s.nz, s.ny, s.nx))
        k = torch.stack(ks)
        F = torch.fft.fftn(E, dim=list(range(-dim, 0)))
        t = torch.einsum("ijmn,jzyx,mnbzyx->ibzyx", C.to(F.dtype), k.to(F.dtype), F)
        A = torch.einsum("ijkl,jzyx,lzyx->zyxik", C, k, k)
        zero = (k * k).sum(0) == 0
        A[zero] = torch.eye(dim, device="cuda", dtype=torch.float64)
        G = torch.linalg.inv(A)
        G[zero] = 0.0
        u = torch.einsum("zyxki,ibzyx->kbzyx", G.to(F.dtype), t)
        ku = torch.einsum("izyx,jbzyx->ijbzyx", k.to(F.dtype), u)
        strain = torch.fft.ifftn(0.5 * (ku + ku.transpose(0, 1)), dim=list(range(-dim, 0))).real
        sig = torch.einsum("ijkl,klbzyx->ijbzyx", C, strain - E)
        return -torch.einsum("ijbzyx,aij->abzyx", sig, e0)

    def trapped(self, P, Pn, U, t):
        """dt times the divergence of the anti-trapping current."""
        s, L, dx = self.s, self.N - 1, self.s.dx
        out = 0.0
        for D, (ax, bc) in enumerate(self.axes()):
            n = P.shape[ax]
            lo, hi = (_padded(P, ax, bc).narrow(ax, o, n + 1) for o in (0, 1))
            rate = _padded(Pn - P, ax, bc)
            rate = 0.5 * (rate.narrow(ax, 0, n + 1) + rate.narrow(ax, 1, n + 1))
            m = _padded(U, ax, bc)
            m = 0.5 * (m.narrow(ax, 0, n + 1) + m.narrow(ax, 1, n + 1))
            pf, both = 0.5 * (lo + hi), lo + hi
            gr = [(hi - lo) / dx if e == D else (_shift(both, a2, 1, b2) - _shift(both, a2, -1, b2)) / (4 * dx)
                  for e, (a2, b2) in enumerate(self.axes())]
            n2 = sum(g * g for g in gr)
            has = n2 >= 1e-12
            inv = torch.where(has, n2.clamp(min=1e-12).rsqrt(), torch.zeros_like(n2))
            pos = self.pos
            if D == self.dim - 1:
                pos = _padded(pos, ax, bc)
                pos = 0.5 * (pos.narrow(ax, 0, n + 1) + pos.narrow(ax, 1, n + 1))
            T = self.temperature(t, pos)
            c = self.composition(m, T)
            J = 0.0
            for a in range(L):
                p = pf[a]
                hp = p * p * (3 - 2 * p)
                inside = (p > 0) & (p < 1)
                root = torch.where(inside, p * (1 - p), torch.ones_like(p)).rsqrt()
                A = torch.where(inside, math.pi / 4 * s.eps * p * (1 - hp) * root, torch.zeros_like(p))
                toward = -sum(g[a] * g[L] for g in gr) * inv[a] * inv[L]
                J = J + (A * rate[a] * gr[D][a] * inv[a] * toward)[None] * (c[a] - c[L])
            out = out + (J.narrow(ax, 1, n) - J.narrow(ax, 0, n)) / dx
        return out

    def composition(self, U, T):
        """c^a_i(mu, T), [N, NM, ...]."""
        y = [U[j][None] - (self.B0[:, j].reshape(-1, 1, 1, 1, 1) + self.B1[:, j].reshape(-1, 1, 1, 1, 1) * T)
             for j in range(self.NM)]
        return torch.stack([sum(self.chi[:, i, j].reshape(-1, 1, 1, 1, 1) * y[j] for j in range(self.NM))
                            for i in range(self.NM)], 1)

    def step(self, P, U, t):
        s, N, NM, dt = self.s, self.N, self.NM, self.dt
        col = lambda v: v.reshape(-1, 1, 1, 1, 1)  # noqa: E731
        T = self.temperature(t, self.pos)
        dev = dict(device=P.device, dtype=P.dtype)
        gam = torch.tensor(s.gamma, **dev)
        if s.potential == "obstacle":
            W = 16 / math.pi ** 2 * torch.einsum("ab,bczyx->aczyx", gam, P)
        else:
            W = 18 * P * torch.einsum("ab,bczyx->aczyx", gam, P * P)
        e1 = P.sum(0)
        e2 = 0.5 * (e1 * e1 - (P * P).sum(0))
        if self.g3:
            W = W + self.g3 * (e2 - P * (e1 - P))
        rate = s.eps * (self.div_flux(P) - self.centre(P)) - W / s.eps
        if not s.grain_growth:
            c = self.composition(U, T)
            psi = []
            for a in range(N):
                y = [U[j] - (self.B0[a, j] + self.B1[a, j] * T) for j in range(NM)]
                C = self.C[0][a] + T * (self.C[1][a] + T * self.C[2][a]) + self.f0[a]
                psi.append(C - 0.5 * sum(c[a, i] * y[i] for i in range(NM)))
            psi = torch.stack([v.expand(P.shape[1:]) for v in psi])
            if s.elastic_C is not None:
                psi = psi + self.elastic(P)
            own = psi * (6 * P - 6 * P * P + 2 * (e2 - P * (e1 - P)))
            S1, S2 = (psi * P).sum(0), (psi * P * P).sum(0)
            rate = rate - own - 2 * ((e1 - P) * (S1 - psi * P) - (S2 - psi * P * P))
        Pn = self.project(P, P + dt * self.mob / s.eps * rate)
        if s.grain_growth:
            return Pn, U
        hn, ho = self.h(Pn), self.h(P)
        DX = torch.einsum("aij,ajk->aik", self.D, self.chi)
        M = torch.einsum("abzyx,aij->ijbzyx", ho, DX)
        div = 0.0
        for ax, bc in self.axes():
            n = P.shape[ax]
            pm, pu = _padded(M, ax, bc), _padded(U, ax, bc)
            flux = (0.5 * (pm.narrow(ax, 0, n + 1) + pm.narrow(ax, 1, n + 1)) *
                    (pu.narrow(ax, 1, n + 1) - pu.narrow(ax, 0, n + 1))[None]).sum(1) / s.dx
            div = div + (flux.narrow(ax, 1, n) - flux.narrow(ax, 0, n)) / s.dx
        rhs = dt * div - (c * (hn - ho)[:, None]).sum(0) - torch.stack([(hn * col(self.dcT[:, i])).sum(0) for i in range(NM)])
        if s.anti_trapping:
            rhs = rhs - self.trapped(P, Pn, U, t)
        X = torch.einsum("abzyx,aij->ijbzyx", hn, self.chi)
        if NM == 1:
            return Pn, U + rhs / X[0]
        det = X[0, 0] * X[1, 1] - X[0, 1] * X[1, 0]
        return Pn, U + torch.stack([(X[1, 1] * rhs[0] - X[0, 1] * rhs[1]) / det, (X[0, 0] * rhs[1] - X[1, 0] * rhs[0]) / det])

    def run(self, P, U, steps):
        for k in range(steps):
            P, U = self.step(P, U, k * self.s.dt)
        return P, U

    def mass(self, P, U, t):
        c = self.composition(U, self.temperature(t, self.pos))
        return [float((self.h(P) * c[:, i]).sum()) for i in range(self.NM)]


def exact(case, seed):
    kind, steps = case["kind"], case["steps"]
    if kind == "sim":
        phases = 8 if case["scene"] in ("multigrain", "grains") else 3
        if case["option"] == "noise" or case["nx"] * case["ny"] * case["nz"] * phases > 7e7:
            return None   # the noise's variates are the library's own; the largest grids take too long
        spec, phi, mu = _sim_inputs(case, seed)
        E = _Exact(spec)
        P, U = E.run(phi.double()[:, None], mu.double()[:, None], steps)
        mass = E.mass(P, U, steps * spec.dt) if case["scene"] in ("deck", "eutectic") else []
        return {"phi": P[:, 0], "mu": U[:, 0], "mass": mass}
    if kind == "sparse":
        spec, phi = _sparse_inputs(case, seed)
        P = phi.double()[:, None]
        P, _ = _Exact(spec, active=True, gamma3=15.0).run(P, P[:1], steps)
        return {"phi": P[:, 0].cpu().numpy()}
    if kind == "batch":
        inputs = _batch_inputs(case, seed)
        phi, mu = [None] * len(inputs), [None] * len(inputs)
        for size in sorted(set(_batch_layout(case))):
            at = [i for i, v in enumerate(_batch_layout(case)) if v == size]
            per = lambda f: torch.tensor([f(inputs[i][0]) for i in at], device="cuda", dtype=torch.float64).reshape(-1, 1, 1, 1)  # noqa: E731
            d = per(lambda s: float(s.delta[0, 1]))
            E = _Exact(inputs[at[0]][0], delta=[[0, d], [d, 0]], f0=[per(lambda s: float(s.f0[0])), 0.0],
                       dt=per(lambda s: s.dt))
            P, U = E.run(torch.stack([inputs[i][1].float().double() for i in at], 1),
                         torch.stack([inputs[i][2].float().double() for i in at], 1), steps)
            for k, i in enumerate(at):
                phi[i], mu[i] = P[:, k].cpu().numpy(), U[:, k].cpu().numpy()
        return {"phi": phi, "mu": mu}
    spec, phi, mu, target = _adjoint_inputs(case, seed)
    t = _types(case)
    phi, mu = phi.to(t).double().requires_grad_(), mu.to(t).double().requires_grad_()
    theta = torch.tensor(theta_of(spec), dtype=t).to("cuda").double().requires_grad_()
    E = _Exact(spec, delta=[[0, theta[0]], [theta[0], 0]], tau=1.0 / theta[1], D=theta[2:].reshape(2, 1, 1))
    P, U = phi[:, None], mu[:, None]
    for k in range(steps):
        P, U = torch.utils.checkpoint.checkpoint(E.step, P, U, k * spec.dt, use_reentrant=False)
    loss = ((P[:, 0] - target.to(t).double()) ** 2).sum()
    dphi, dmu, dtheta = torch.autograd.grad(loss, (phi, mu, theta))
    return {"phi": P[:, 0].detach(), "mu": U[:, 0].detach(), "dphi": dphi, "dmu": dmu, "dtheta": dtheta}
