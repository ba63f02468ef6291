"""Performance cases: what a user of the library has it compute, through its
public binding (``paper_1810_08572_gb300.fvs``), over the range of sizes and
options that the configurations, tests and benchmark of this repository use.

A case is a dict of plain values; ``prepare`` makes what a program holds
before the call (mesh, solver or model, inputs on the GPU), ``run`` makes one
pass and returns everything the pass computes.

Stepping cases run with solver tolerances tight enough that the fields that
come back are those of the discrete equations to about ten digits, as the
repository's parity tests do, and not the point where an iteration stopped.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from fvs_inputs import box_mesh, cases, casting_mesh
from paper_1810_08572_gb300 import fvs

TIGHT = dict(p_rtol=1e-12, mom_rtol=1e-12, e_rtol=1e-13, e_tol_T=1e-10, max_krylov_iters=2000)
FIELDS = ("T", "FS", "U", "P", "FLUX")

# conductivity of the metal falling with temperature (piecewise linear), and
# the film of a cooled die, as in the tests of those options
K_TABLE = [(600.0, 190.0), (833.0, 160.0), (913.0, 110.0), (1000.0, 100.0)]
FILM = [(2, 600.0, 3000.0), (2, 600.0, 1500.0), (0, 0.0), (2, 550.0, 800.0), (0, 0.0), (0, 0.0)]

UQ_FAMILIES = (0, 1, 1)        # melt temperature normal, wall temperature and solute uniform
UQ_PARAMS = ((950.0, 10.0), (650.0, 750.0), (3.0, 5.0))


def listed():
    return [
        # the smallest transient a user runs: a 32 x 32 x 4 orthogonal cavity
        # (4,096 cells), launches and host round trips count
        dict(name="step_cavity_4k", kind="step", nx=32, ny=32, nz=4, jitter=0.0, precision=0, steps=20, front=0.8,
             physics="flow"),
        # an odd, ragged, skewed mesh of middling size in FP64
        dict(name="step_plate_odd", kind="step", nx=83, ny=61, nz=19, jitter=0.2, precision=0, steps=6, front=0.7,
             physics="flow"),
        # the benchmark's mesh: 128^3 jittered and renumbered, all melt, FP64
        dict(name="step_cavity_128", kind="step", nx=128, ny=128, nz=128, jitter=0.2, precision=0, steps=3, front=1.0,
             physics="flow"),
        # a front half way through the casting, mixed precision: cells freeze
        # and melt again in every step, the hierarchy is refreshed
        dict(name="step_front_96_mixed", kind="step", nx=96, ny=96, nz=96, jitter=0.2, precision=1, steps=4,
             front=0.55, physics="flow"),
        # plate with ribs and riser in its steel mold, 1 mm voxels (615,176
        # cells), mixed precision
        dict(name="step_casting_mold", kind="casting", h=1e-3, precision=1, steps=5),
        # castings without natural convection: Scheil alloy, k(T), film-cooled walls
        dict(name="step_conduction", kind="step", nx=72, ny=64, nz=40, jitter=0.2, precision=0, steps=8, front=0.6,
             physics="conduction"),
        # the pressure system alone on an orthogonal mesh (AMG-CG)
        dict(name="pressure_solve", kind="pressure", nx=96, ny=96, nz=48, precision=0),
        # first steps of a batch of uncertain samples in lockstep, mixed precision
        dict(name="uq_lockstep", kind="uq", nx=24, ny=24, nz=8, samples=32, steps=20, precision=1),
        # training the network surrogate on 512 solves (100 of its epochs)
        dict(name="surrogate_train", kind="train", rows=512, epochs=100),
        # a handful of samples asked of the network from the host
        dict(name="surrogate_query", kind="predict", rows=1000, device=False),
        # Monte Carlo on the network, a million samples
        dict(name="surrogate_monte_carlo", kind="predict", rows=1000000, device=True),
        # Monte Carlo on the polynomial chaos, a million samples
        dict(name="pce_monte_carlo", kind="pce", rows=1000000, degree=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "casting", "pressure", "uq", "train", "predict", "predict", "pce"])
    if kind == "step":
        nx, ny = _log(rng, 16, 128), _log(rng, 16, 128)
        nz = min(_log(rng, 4, 128), max(4, 1200000 // (nx * ny)))
        physics = rng.choice(["flow", "flow", "flow", "conduction"])
        return dict(kind="step", nx=nx, ny=ny, nz=nz, jitter=rng.choice([0.0, 0.2]), precision=rng.randrange(2),
                    steps=rng.randint(2, 5), front=rng.choice([1.0, round(rng.uniform(0.4, 0.95), 3)]),
                    physics=physics)
    if kind == "casting":
        return dict(kind="casting", h=round(rng.uniform(1.0e-3, 2.5e-3), 6), precision=rng.randrange(2),
                    steps=rng.randint(2, 5))
    if kind == "pressure":
        return dict(kind="pressure", nx=_log(rng, 16, 112), ny=_log(rng, 16, 112), nz=_log(rng, 4, 64),
                    precision=rng.randrange(2))
    if kind == "uq":
        return dict(kind="uq", nx=rng.randint(8, 24), ny=rng.randint(8, 24), nz=rng.randint(4, 12),
                    samples=rng.randint(5, 48), steps=rng.randint(4, 16), precision=rng.randrange(2))
    if kind == "train":
        return dict(kind="train", rows=_log(rng, 60, 2048), epochs=rng.randint(20, 100))
    if kind == "predict":
        return dict(kind="predict", rows=_log(rng, 1, 2000000), device=rng.random() < 0.7)
    return dict(kind="pce", rows=_log(rng, 100, 2000000), degree=rng.randint(2, 7))


# --------------------------------------------------------------------------
# what a program has in hand
# --------------------------------------------------------------------------
@functools.lru_cache(maxsize=24)
def _box(nx, ny, nz, jitter):
    """Mesh lists of the cavity; skewed meshes are renumbered at random, as the benchmark's is."""
    if jitter > 0:
        return box_mesh(nx, ny, nz, cases.CAVITY, jitter=jitter, jitter_seed=1810, permute_seed=8572)
    return box_mesh(nx, ny, nz, cases.CAVITY)


@functools.lru_cache(maxsize=8)
def _casting(h):
    return casting_mesh(h)


def _waves(x, seed, amplitude):
    """A smooth field of random phase and size over the unit box (x: [n, 3])."""
    rng = np.random.default_rng(seed)
    out = torch.zeros(x.shape[0], dtype=torch.float64, device="cuda")
    for a in rng.integers(1, 4, size=(6, 3)):
        ph, c = rng.uniform(0, 2 * np.pi, 3), rng.uniform(0.4, 1.0)
        w = torch.full_like(out, float(c))
        for d in range(3):
            w = w * torch.cos(math.pi * float(a[d]) * x[:, d] + float(ph[d]))
        out += w
    return amplitude / 2.5 * out


def _unit(mesh):
    n = torch.tensor(mesh["shape"], dtype=torch.float64, device="cuda")
    return (torch.from_numpy(mesh["cell_ijk"]).cuda().double() + 0.5) / n


def _profile(x, front, seed):
    """Melt freezing from the cold wall at x = 0: the 1-D conduction profile
    that puts the solidus at 1 - front of the length, plus slow waves of a few
    kelvin (all melt for front = 1)."""
    if front >= 1.0:
        return 945.0 + _waves(x, seed, 8.0)
    z = 0.5079        # erf(z) = 133/250: T = 833 K there
    T = 700.0 + 250.0 * torch.special.erf(x[:, 0] * z / (1.0 - front))
    return T + _waves(x, seed, 3.0)


def _props(case):
    if case["physics"] == "conduction":
        return cases.props(material=cases.AL_SI_SCHEIL, walls=FILM, T_init=950.0, precision=case["precision"],
                           no_flow=True, k_table=K_TABLE, **TIGHT)
    return cases.props(precision=case["precision"], **TIGHT)


def _solver_state(mesh, props, T):
    stream = torch.cuda.Stream()
    M = fvs.Mesh(mesh, stream=stream)
    S = fvs.Solver(M, props, stream=stream)
    nc, nf = M.n_cells, M.n_faces
    size = dict(T=nc, FS=nc, U=3 * nc, P=nc, FLUX=nf)
    out = {f: torch.zeros(size[f], dtype=torch.float64, device="cuda") for f in FIELDS}
    torch.cuda.synchronize()
    return dict(mesh=M, solver=S, T=T, out=out)


def prepare(case, seed):
    k = case["kind"]
    if k == "step":
        m = _box(case["nx"], case["ny"], case["nz"], case["jitter"])
        s = _solver_state(m, _props(case), _profile(_unit(m), case["front"], seed))
    elif k == "casting":
        m = _casting(case["h"])
        x = _unit(m)
        w = _waves(x, seed, 10.0)
        mold = torch.from_numpy(m["cell_zone"]).cuda() == 1
        T = torch.where(mold, 520.0 + w, 935.0 + w)
        s = _solver_state(m, cases.casting_props(precision=case["precision"], **TIGHT), T)
    elif k == "pressure":
        m = _box(case["nx"], case["ny"], case["nz"], 0.0)
        s = _solver_state(m, cases.props(precision=case["precision"], **TIGHT), None)
        s["solver"].step(1e-3)          # the active set of the solve: all melt
        s["rhs"] = _pressure_rhs(case, seed)
        s["p"] = torch.zeros_like(s["rhs"])
    elif k == "uq":
        m = _box(case["nx"], case["ny"], case["nz"], 0.0)
        s = dict(mesh=fvs.Mesh(m), props=cases.props(precision=case["precision"], **TIGHT),
                 X=cases.uq_inputs(case["samples"], seed))
    elif k == "train":
        X, Y = _training_set(case["rows"], seed)
        s = dict(X=X, Y=Y, seed=seed % 1000)
    elif k == "predict":
        S, X = _network(case, seed)
        s = dict(model=S, X=X)
        if case["device"]:
            s["X"] = torch.from_numpy(X).cuda()
            s["Y"] = torch.zeros(case["rows"], 4, dtype=torch.float64, device="cuda")
    else:
        P, X = _chaos(case, seed)
        s = dict(model=P, X=torch.from_numpy(X).cuda(),
                 Y=torch.zeros(case["rows"], 4, dtype=torch.float64, device="cuda"))
    s.update(kind=k, case=dict(case))
    return s


def _pressure_rhs(case, seed):
    """Right side of the pressure equation with zero sum: smooth waves and noise."""
    m = _box(case["nx"], case["ny"], case["nz"], 0.0)
    g = torch.Generator(device="cuda").manual_seed(seed)
    n = len(m["cells"])
    b = _waves(_unit(m), seed, 1.0) + 0.3 * torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
    vol = math.prod(cases.CAVITY) / n
    return (b - b.mean()) * vol


def _response(X):
    """Smooth stand-ins of the four outputs (solidification time, cooling
    rate, arm spacing, yield strength) over the uncertain inputs."""
    tm, tw, c = ((X - np.array([950.0, 700.0, 4.0])) / np.array([10.0, 30.0, 0.6])).T
    t = 0.55 + 0.012 * tm + 0.11 * tw - 0.04 * c + 0.02 * tw * tw - 0.004 * tm * tw
    t = np.abs(t) + 0.05
    cr = 80.0 / t
    lam = 39.4 * cr ** -0.317
    return np.stack([t, cr, lam, 59.0 / np.sqrt(lam) + 120.3], axis=1)


def _training_set(rows, seed):
    X = cases.uq_inputs(rows, seed)
    Y = _response(X)
    return X, Y * (1.0 + 0.003 * np.random.default_rng(seed + 1).standard_normal(Y.shape))


SIZES = (3, 128, 128, 128, 128, 4)


def _network_params(seed):
    """Weights of the size a trained network has, flattened per layer: W row-major, then b."""
    rng = np.random.default_rng(seed + 7)
    return [(rng.standard_normal((b, a)) * math.sqrt(1.6 / a), 0.2 * rng.standard_normal(b))
            for a, b in zip(SIZES[:-1], SIZES[1:])]


SCALE = (np.array([950.0, 700.0, 4.0]), np.array([10.0, 29.0, 0.58]),
         np.array([0.6, 150.0, 8.0, 141.0]), np.array([0.1, 25.0, 0.4, 0.6]))


def _network(case, seed):
    S = fvs.Surrogate(3, 128, 4, 4, seed=1)
    S.set_scaling(*SCALE)
    S.set_params(np.concatenate([np.concatenate([W.ravel(), b]) for W, b in _network_params(seed)]))
    return S, cases.uq_inputs(case["rows"], seed)


def _chaos(case, seed):
    P = fvs.Pce(UQ_FAMILIES, UQ_PARAMS, case["degree"], 4)
    Xt, Yt = _training_set(512, seed)
    P.fit(Xt, Yt)
    return P, cases.uq_inputs(case["rows"], seed + 3)


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def run(state):
    k = state["kind"]
    if k in ("step", "casting"):
        # a transient from a given state: some steps, then the fields
        S, out = state["solver"], state["out"]
        S.set_state(state["T"])
        S.step(1e-3, state["case"]["steps"])
        for f in FIELDS:
            S.query(f, out=out[f])
        return out
    if k == "pressure":
        state["solver"].pressure_solve(state["rhs"], state["p"], TIGHT["p_rtol"])
        return state["p"]
    if k == "uq":
        qoi, steps, extra = fvs.uq_run(state["mesh"], state["props"], state["X"], 2e-3, state["case"]["steps"],
                                       fields=True)
        return dict(qoi=qoi, steps=steps, T=extra["T"], U=extra["U"], P=extra["P"])
    if k == "train":
        X, Y = state["X"], state["Y"]
        S = fvs.Surrogate(3, 128, 4, 4, seed=state["seed"])
        S.set_scaling(X.mean(0), X.std(0), Y.mean(0), Y.std(0))
        loss = S.train(X, Y, state["case"]["epochs"], 1e-3)
        return dict(params=S.get_params(), loss=loss)
    if k == "predict":
        if state["case"]["device"]:
            return state["model"].predict(state["X"], out=state["Y"])
        return state["model"].predict(state["X"])
    return state["model"](state["X"], out=state["Y"])


# --------------------------------------------------------------------------
# what a pass cannot do without, and its values in 64 bits
# --------------------------------------------------------------------------
def work(case):
    k = case["kind"]
    if k in ("step", "casting", "uq"):
        if k == "casting":
            n = 0.000615176 / case["h"] ** 3          # cells of the 1 mm casting, scaled
            w = 7
        else:
            n = case["nx"] * case["ny"] * case["nz"]
            w = 27 if case.get("jitter", 0.0) > 0 else 7
        samples = case.get("samples", 1)
        flow = 0 if case.get("physics") == "conduction" else 1
        # per step: the operators of momentum, pressure and energy once, the
        # fields of two time levels read and those of the next written
        # (T, fs, u, p per cell, a flux per face)
        op = (1 + 2 * flow) * w * 12.0 * n
        fields = 8.0 * n * (3 * 3 + flow * (3 * 3 + 2 + 3 * 3))
        return dict(bytes=case["steps"] * (op + samples * fields),
                    flops=case["steps"] * samples * n * (1 + 4 * flow) * 2.0 * w * 2)
    if k == "pressure":
        n = case["nx"] * case["ny"] * case["nz"]
        return dict(bytes=n * (7 * 12.0 + 16.0), flops=n * 28.0)
    weights = sum(a * b for a, b in zip(SIZES[:-1], SIZES[1:]))
    if k == "train":
        return dict(bytes=56.0 * case["rows"] + 24.0 * weights, flops=6.0 * weights * case["rows"] * case["epochs"])
    if k == "predict":
        return dict(bytes=56.0 * case["rows"] + 2.0 * weights, flops=2.0 * weights * case["rows"])
    terms = math.comb(case["degree"] + 3, 3)
    return dict(bytes=56.0 * case["rows"] + 32.0 * terms, flops=2.0 * terms * 4 * case["rows"])


def _gelu(z):
    return 0.5 * z * (1.0 + torch.special.erf(z / math.sqrt(2.0)))


def exact(case, seed):
    k = case["kind"]
    if k == "pressure":
        # uniform box, no-flux walls: the cosine transform diagonalises the system
        b = _pressure_rhs(case, seed)
        n = (case["nz"], case["ny"], case["nx"])
        h = [L / m for L, m in zip(reversed(cases.CAVITY), n)]
        area = [h[1] * h[2], h[0] * h[2], h[0] * h[1]]
        C, lam = [], []
        for d in range(3):
            i = torch.arange(n[d], dtype=torch.float64, device="cuda")
            c = torch.cos(math.pi / n[d] * (i[None, :] + 0.5) * i[:, None]) * math.sqrt(2.0 / n[d])
            c[0] /= math.sqrt(2.0)
            C.append(c)
            lam.append(4.0 * area[d] / h[d] * torch.sin(0.5 * math.pi * i / n[d]) ** 2)
        t = torch.einsum("ka,lb,mc,abc->klm", *C, b.reshape(n))
        e = lam[0][:, None, None] + lam[1][None, :, None] + lam[2][None, None, :]
        e[0, 0, 0] = 1.0
        t = -cases.AL_ALLOY["rho"] * t / e
        t[0, 0, 0] = 0.0
        return torch.einsum("ka,lb,mc,klm->abc", *C, t).reshape(-1)
    if k == "predict":
        mu, sd, mo, so = (torch.from_numpy(a).cuda() for a in SCALE)
        h = (torch.from_numpy(cases.uq_inputs(case["rows"], seed)).cuda() - mu) / sd
        layers = _network_params(seed)
        for i, (W, b) in enumerate(layers):
            h = h @ torch.from_numpy(W).cuda().T + torch.from_numpy(b).cuda()
            if i < len(layers) - 1:
                h = _gelu(h)
        return h * so + mo
    if k == "pce":
        Xt, Yt = _training_set(512, seed)
        c = torch.from_numpy(np.linalg.lstsq(_vandermonde(Xt, case["degree"]).numpy(), Yt, rcond=None)[0])
        X = cases.uq_inputs(case["rows"], seed + 3)
        return torch.cat([_vandermonde(X[i:i + 100000], case["degree"]) @ c for i in range(0, len(X), 100000)])
    return None


def _vandermonde(X, p):
    """Products of orthonormal Hermite (melt temperature) and Legendre polynomials up to total degree p."""
    X = torch.from_numpy(np.asarray(X))
    B = []
    for j, (fam, (a, b)) in enumerate(zip(UQ_FAMILIES, UQ_PARAMS)):
        xi = (X[:, j] - a) / b if fam == 0 else (2.0 * X[:, j] - a - b) / (b - a)
        v = [torch.ones_like(xi), xi]
        for n in range(1, p):
            v.append(xi * v[n] - n * v[n - 1] if fam == 0 else ((2 * n + 1) * xi * v[n] - n * v[n - 1]) / (n + 1))
        B.append([q / math.sqrt(math.factorial(n)) if fam == 0 else q * math.sqrt(2 * n + 1)
                  for n, q in enumerate(v)])
    return torch.stack([B[0][i] * B[1][j] * B[2][l] for i in range(p + 1) for j in range(p + 1 - i)
                        for l in range(p + 1 - i - j)], dim=1)
