"""What a program does with this framework, as timed cases through its public entry points.

A case names a kind of work and its sizes; inputs (sources, conductivities, initial factors,
points, training data) come from the seed.  The kinds:

  solve      Problem.solve at a fixed number of modes and sweeps from seeded random factors:
             the subspace iteration with its residuals, on every reduced solver
  setup      the same from the bare description: assembly, sources, decompositions, solve
  batch      Batch.sweep over independent instances of different dims, sizes and mode counts
  nonlinear  GlobalLocal.solve: global stages with solution-dependent coefficients
  grid       Problem.eval_grid on (strided) node slices, FP32 and FP64
  points     Problem.eval_points at scattered points
  mlp        the warm-start network: training steps, or one forward pass

Sources are sums of as many separable Gaussians as there are modes (and two more), as for a
plate under many heat sources, so that the factors have full rank and the outputs of a solve
are determined to rounding; the laser cases bring the moving source's own terms.
"""
import functools
import math

import numpy as np
import torch

from paper_2503_13933_gb300 import nonlinear, taps
from paper_2503_13933_gb300 import workloads as W

SOLVERS = {"block": taps.SOLVER_BLOCK_LU, "fastdiag": taps.SOLVER_FASTDIAG, "modediag": taps.SOLVER_MODEDIAG}


def listed():
    return [
        # the smallest solve: a coarse box, a few modes, the default solver; calls and launches count
        dict(name="solve_box_16", kind="solve", family="poisson", D=3, n=16, M=4, solver="block", sweeps=2),
        # the plain FP64 configuration, 64 nodes per dim, on the default solver
        dict(name="solve_plain_64", kind="solve", family="poisson", D=3, n=64, M=10, solver="block", sweeps=2),
        # the headline space-parameter problem: 3D space and the conductivity as a fourth dim
        dict(name="solve_space_parameter", kind="solve", family="poisson_k", n=256, n_par=32, M=30,
             solver="fastdiag", sweeps=3),
        # the powder-bed-fusion slab: moving source, convection faces, a time dim, three parameters
        dict(name="solve_slab", kind="solve", family="slab", n=256, n_z=64, n_t=64, n_par=16, M=20,
             solver="fastdiag", sweeps=2),
        # the large moving-source configuration at 100 modes
        dict(name="solve_large", kind="solve", family="large", n=1536, n_t=256, n_par=16, M=100,
             solver="fastdiag", sweeps=1),
        # the headline problem from its description to its factors on the host, nothing kept
        dict(name="setup_and_solve", kind="setup", family="poisson_k", n=256, n_par=32, M=30, solver="fastdiag",
             sweeps=3),
        # independent instances of mixed size swept together
        dict(name="batch_sweep", kind="batch", count=24, n_lo=32, n_hi=512, M_lo=4, M_hi=32, layout=4000, sweeps=2),
        # a plate whose heat capacity and conductivity depend on the temperature: weighted operators
        dict(name="nonlinear_stage", kind="nonlinear", n=64, n_z=11, n_t=64, M=6, sweeps=2, stages=2),
        # the whole space-parameter field in FP32
        dict(name="grid_field_f32", kind="grid", D=4, n=256, n_last=32, M=30, step=1, dtype="f32"),
        # a strided FP64 slice with odd sizes
        dict(name="grid_slice_f64", kind="grid", D=4, n=203, n_last=23, M=17, step=2, dtype="f64"),
        # the error estimate of the eight-dimensional study: the field at scattered points
        dict(name="points_8d", kind="points", D=8, n=128, M=8, count=65536),
        # training the warm-start network on sixteen instances of 30 modes
        dict(name="mlp_train", kind="mlp", n_in=21, hidden=256, layers=3, n_out=257, batch=480, steps=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "setup", "batch", "nonlinear", "grid", "grid", "points", "mlp"])
    if kind in ("solve", "setup"):
        family = rng.choice(["poisson", "poisson_k", "heat", "slab"] if kind == "solve" else ["poisson", "poisson_k"])
        if family == "slab":
            return dict(kind="solve", family="slab", n=_log(rng, 48, 384), n_z=rng.randint(24, 96),
                        n_t=rng.randint(24, 96), n_par=rng.randint(8, 16), M=rng.randint(4, 24), solver="fastdiag",
                        sweeps=rng.randint(1, 2))
        solver = "fastdiag" if kind == "setup" else rng.choice(["block", "fastdiag", "fastdiag", "modediag"])
        wide = solver == "fastdiag"
        c = dict(kind=kind, family=family, n=_log(rng, 16, 384 if wide else 128),
                 M=_log(rng, 3, 64 if wide and kind == "solve" and family == "poisson_k" else 32 if wide else 16),
                 solver=solver, sweeps=rng.randint(1, 3))
        if family == "poisson":
            c["D"] = rng.randint(3, 5)
        else:
            c["n_par"] = rng.randint(12, 48)
        return c
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(4, 24), n_lo=32, n_hi=_log(rng, 64, 512), M_lo=4,
                    M_hi=rng.randint(8, 32), layout=rng.randrange(1000), sweeps=rng.randint(1, 3))
    if kind == "nonlinear":
        return dict(kind="nonlinear", n=rng.randint(24, 96), n_z=rng.randint(9, 15), n_t=rng.randint(24, 80),
                    M=rng.randint(3, 8), sweeps=2, stages=2)
    if kind == "grid":
        dtype = rng.choice(["f32", "f64"])
        c = dict(kind="grid", D=rng.randint(3, 5), n=rng.randint(20, 180), n_last=rng.randint(5, 40),
                 M=_log(rng, 3, 100), step=rng.randint(1, 3), dtype=dtype)
        most = 4e8 if dtype == "f32" else 3e7   # values of the field
        while np.prod([float(dm["n"] // c["step"] + 1) for dm in _grid_description(c)["dims"]]) > most:
            c["n"] = c["n"] * 3 // 4
        return c
    if kind == "points":
        return dict(kind="points", D=rng.randint(3, 8), n=_log(rng, 16, 450), M=_log(rng, 3, 32),
                    count=_log(rng, 1000, 200000))
    return dict(kind="mlp", n_in=rng.randint(2, 24), hidden=rng.choice([64, 128, 200, 256]), layers=rng.randint(2, 4),
                n_out=rng.randint(65, 400), batch=_log(rng, 30, 1600), steps=rng.choice([0, 5, 10]))


# ---------------------------------------------------------------------------------
# Descriptions: the seeded inputs as plain data (dims, terms, sources)
# ---------------------------------------------------------------------------------
def _bumps(rng, dims, count, tail):
    """`count` separable Gaussians over the first dims, `tail` for the factors of the others."""
    out = []
    for _ in range(count):
        amp, facs = float(rng.uniform(0.5, 2.0)), []
        for dm in dims[:len(dims) - len(tail)]:
            L = dm["hi"] - dm["lo"]
            facs.append(("gauss", (dm["lo"] + float(rng.uniform(0.1, 0.9)) * L, float(rng.uniform(0.03, 0.15)) * L)))
        out.append((amp, facs + [f(rng) for f in tail]))
    return out


def _poisson(ns, M, seed, transient=False):
    rng = np.random.default_rng(seed)
    D = len(ns)
    dims = [W.dim(n) for n in ns]
    ops = [["K" if d == e else "M" for d in range(D)] for e in range(D)]
    tail = []
    if transient:
        dims[-1] = W.dim(ns[-1], kind=W.TIME, dirichlet_lo=True, dirichlet_hi=False)
        ops = [["M"] * (D - 1) + ["G"]] + [o[:-1] + ["M"] for o in ops[:-1]]
        # each source is switched on and off in its own window of time
        tail = [lambda r: ("gauss", (float(r.uniform(0.1, 0.9)), float(r.uniform(0.05, 0.2))))]
    return dict(name="poisson", dims=dims, terms=[(1.0, o) for o in ops],
                sources=_bumps(rng, dims, M + 2, tail))


@functools.lru_cache(maxsize=4)
def _laser(family, n, n_z, n_t, n_par):
    if family == "slab":
        return W.lpbf_slab(n_xy=n, n_z=n_z, n_t=n_t, n_par=n_par)
    return W.lpbf_large(n_xy=n, n_z=n, n_t=n_t, n_par=n_par)


def _describe(case, seed):
    f, n, M = case["family"], case["n"], case["M"]
    if f == "poisson":
        return _poisson([n] * case["D"], M, seed)
    if f == "heat":
        return _poisson([n] * 3 + [case["n_par"]], M, seed, transient=True)
    rng = np.random.default_rng(seed)
    if f == "poisson_k":
        desc = W.poisson_k(n_space=n, n_k=case["n_par"], seed=seed)
        # every source carries its own conductivity dependence
        tail = [lambda r: ("gauss", (float(r.uniform(1.0, 10.0)), float(r.uniform(1.0, 4.0))))]
        return dict(desc, sources=_bumps(rng, desc["dims"], M + 2, tail))
    base = _laser(f, n, case.get("n_z", 0), case["n_t"], case["n_par"])
    # another material: the diffusion terms' conductivity and the absorbed power
    k, eta = float(rng.uniform(0.8, 1.2)), float(rng.uniform(0.8, 1.2))
    terms = [(a * k if "K" in ops else a, ops) for a, ops in base["terms"]]
    return dict(base, terms=terms, sources=[(b * eta, facs) for b, facs in base["sources"]])


def _batch_layout(case):
    """Per instance its sizes, mode count and whether its last dim is time: from the case alone."""
    rng = np.random.default_rng(case["layout"])
    out = []
    for _ in range(case["count"]):
        D = int(rng.integers(3, 6))
        ns = [int(v) for v in rng.integers(case["n_lo"], case["n_hi"] + 1, size=D)]
        out.append((ns, int(rng.integers(case["M_lo"], case["M_hi"] + 1)), bool(rng.integers(0, 2))))
    return out


def _random_factors(desc, M, seed):
    rng = np.random.default_rng([seed, 1])
    return [rng.uniform(-1.0, 1.0, (W.n_free(dm), M)) for dm in desc["dims"]]


def _plate(case, seed):
    # an 11-element-deep plate under several fixed sources with their own time windows
    rng = np.random.default_rng(seed)
    base = W.nonlinear_track(n_xy=case["n"], n_z=case["n_z"], n_t=case["n_t"])
    T = base["dims"][3]["hi"]
    tail = [lambda r: ("gauss", (T * float(r.uniform(0.2, 0.9)), T * float(r.uniform(0.1, 0.3))))]
    return dict(base, sources=[(50.0 * b, f) for b, f in _bumps(rng, base["dims"], case["M"] + 2, tail)])


def _grid_description(case):
    D, n = case["D"], case["n"]
    ns = [n] * 3 + [case["n_last"]] * (D - 3) if D > 3 else [n, n, case["n_last"]]
    return _poisson(ns, 1, 0)


def _slices(case, desc):
    start = [1 % case["step"] for _ in desc["dims"]]
    count = [(dm["n"] - 1 - s) // case["step"] + 1 for s, dm in zip(start, desc["dims"])]
    return start, count, [case["step"]] * len(count)


# ---------------------------------------------------------------------------------
# What a program has in hand, one pass, and its work
# ---------------------------------------------------------------------------------
class _DeviceArray:
    """The factor matrix of one dim where the library keeps it (column-major, FP64).  A tensor
    made from this object refers to it, and through it to the factors that own the memory."""

    def __init__(self, factors, d, n, M):
        self.factors = factors
        ptr = taps.lib().taps_factors_device_ptr(factors.handle, d)
        self.__cuda_array_interface__ = dict(shape=(M, n), typestr="<f8", data=(ptr, False), version=3, strides=None)


def _views(P, U, M):
    return [torch.as_tensor(_DeviceArray(U, d, n, M), device="cuda") for d, n in enumerate(P.n_free)]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        P = taps.Problem(_describe(case, seed))
        U = P.factors(case["M"])
        return dict(case=case, seed=seed, P=P, U=U, views=_views(P, U, case["M"]))
    if kind == "setup":
        return dict(case=case, seed=seed, desc=_describe(case, seed))
    if kind == "batch":
        Ps, Us, U0s, views, cache = [], [], [], [], []
        for i, (ns, M, transient) in enumerate(_batch_layout(case)):
            desc = _poisson(ns, M, [seed, i], transient)
            stream = torch.cuda.Stream()
            cache.append(stream)
            P = taps.Problem(desc, stream=taps.ctypes.c_void_p(stream.cuda_stream))
            U, U0 = P.factors(M), P.factors(M)
            U0.set(_random_factors(desc, M, seed + i))
            U.copy_from(U0)
            Ps.append(P), Us.append(U), U0s.append(U0)
            views.append(_views(P, U, M))
        B = taps.Batch(Ps, Us, solver=taps.SOLVER_FASTDIAG)
        return dict(case=case, B=B, P=Ps, U=Us, U0=U0s, views=views, streams=cache)
    if kind == "nonlinear":
        desc = _plate(case, seed)
        return dict(case=case, G=nonlinear.GlobalLocal(desc, W.INCONEL_LAW, case["M"]),
                    U0=_random_factors(desc, case["M"], seed))
    if kind == "grid":
        desc = _grid_description(case)
        P = taps.Problem(desc)
        U = P.factors(case["M"])
        U.set(_random_factors(desc, case["M"], seed))
        start, count, step = _slices(case, desc)
        out = torch.empty(count, dtype=torch.float32 if case["dtype"] == "f32" else torch.float64, device="cuda")
        return dict(case=case, P=P, U=U, slices=(start, count, step), out=out)
    if kind == "points":
        desc = _poisson([case["n"]] * case["D"], 1, 0)
        P = taps.Problem(desc)
        U = P.factors(case["M"])
        U.set(_random_factors(desc, case["M"], seed))
        pts = torch.tensor(np.random.default_rng(seed).uniform(0.0, 1.0, (case["count"], case["D"])), device="cuda")
        return dict(case=case, P=P, U=U, pts=pts, out=torch.empty(case["count"], dtype=torch.float64, device="cuda"))
    net = taps.MLP(case["n_in"], case["hidden"], case["layers"], case["n_out"], seed=seed & 0xFFFF)
    params, x, t = _mlp_inputs(case, seed)
    net.set_params(params)
    x, t = torch.tensor(x, device="cuda"), torch.tensor(t, device="cuda")
    return dict(case=case, net=net, x=x, t=t, y=torch.empty_like(t))


def _solve(P, U, case, seed):
    r = P.solve(U, M0=case["M"], M_max=case["M"], als_tol=0.0, res_tol=0.0, max_sweeps=case["sweeps"],
                init=taps.INIT_RANDOM, seed=seed & 0xFFFFFF, solver=SOLVERS[case["solver"]])
    return dict(rho=r["rho"], rho_full=r["rho_full"], change=r["change"])


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        rep = _solve(state["P"], state["U"], case, state["seed"])
        return dict(rep, factors=state["views"])
    if kind == "setup":
        P = taps.Problem(state["desc"])
        U = P.factors(case["M"])
        rep = _solve(P, U, case, state["seed"])
        return dict(rep, factors=U.get())
    if kind == "batch":
        for U, U0 in zip(state["U"], state["U0"]):
            U.copy_from(U0)
        changes = state["B"].sweep(case["sweeps"])
        # the batch has been waited for: the factors of all instances, by mode
        return dict(changes=changes, factors=[torch.cat([v.reshape(-1) for v in vs]) for vs in state["views"]])
    if kind == "nonlinear":
        U, hist = state["G"].solve(case["sweeps"], max_iters=case["stages"], tol=0.0, U0=state["U0"])
        return dict(factors=U, changes=np.array(hist[1:]))
    if kind == "grid":
        return state["P"].eval_grid(state["U"], *state["slices"], state["out"],
                                    dtype=taps.FP32 if case["dtype"] == "f32" else taps.FP64)
    if kind == "points":
        return state["P"].eval_points(state["U"], state["pts"], state["out"])
    if case["steps"]:
        loss = state["net"].train(state["x"], state["t"], case["steps"], lr=1e-3)
        return dict(loss=np.float32(loss), params=state["net"].params())
    return state["net"].forward(state["x"], state["y"])


def work(case):
    kind = case["kind"]
    if kind in ("solve", "setup"):
        return _solve_work(_describe(case, 0), case["M"], case["sweeps"])
    if kind == "batch":
        parts = [_solve_work(_poisson(ns, M, 0, tr), M, case["sweeps"]) for ns, M, tr in _batch_layout(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if kind == "nonlinear":
        desc = _plate(case, 0)
        M, laws = case["M"], 2
        w = _solve_work(dict(desc, terms=[(1.0, ["K"] * 4)]), M, case["sweeps"] * case["stages"])
        # every dim holds its plain operators and one or two weighted ones per mode
        ops = sum(dm["n"] * 11.0 * (2 + laws * M) for dm in desc["dims"])
        return dict(bytes=w["bytes"] + 8.0 * ops, flops=w["flops"] + 2.0 * ops * M * case["sweeps"] * case["stages"])
    if kind == "grid":
        desc = _grid_description(case)
        _, count, _ = _slices(case, desc)
        size = float(np.prod(count))
        esz = 4 if case["dtype"] == "f32" else 8
        return dict(bytes=esz * size + 8.0 * sum(count) * case["M"], flops=2.0 * size * case["M"])
    if kind == "points":
        c, D = case["count"], case["D"]
        return dict(bytes=8.0 * (c * (D + 1) + D * case["n"] * case["M"]), flops=2.0 * c * D * case["M"] * 7)
    dims = [case["n_in"]] + [case["hidden"]] * case["layers"] + [case["n_out"]]
    params = sum(a * b + b for a, b in zip(dims, dims[1:]))
    steps, passes = max(case["steps"], 1), 6.0 if case["steps"] else 2.0
    io = 4.0 * case["batch"] * (case["n_in"] + case["n_out"])
    return dict(bytes=io + 4.0 * params * (2 if case["steps"] else 1), flops=passes * params * case["batch"] * steps)


def _solve_work(desc, M, sweeps):
    """Bands, source vectors and factors once; per sweep and dim the reduced system in its
    cheapest form (one M x M system per node), its contractions and its residual."""
    Rf, by, fl = len(desc["sources"]), 0.0, 0.0
    for d, dm in enumerate(desc["dims"]):
        n = W.n_free(dm)
        ops = len({t[1][d] for t in desc["terms"]})
        by += 8.0 * (ops * n * 11 + Rf * n + n * M)
        fl += n * (2.0 / 3.0 * M ** 3 + 2.0 * M * M) + 2.0 * (2 * ops * n * M * (M + 11) + 2 * Rf * n * M)
    return dict(bytes=by, flops=fl * sweeps)


def _mlp_inputs(case, seed):
    rng = np.random.default_rng([seed, 2])
    dims = [case["n_in"]] + [case["hidden"]] * case["layers"] + [case["n_out"]]
    p = []
    for a, b in zip(dims, dims[1:]):
        p += [rng.uniform(-1, 1, a * b) * math.sqrt(6.0 / (a + b)), np.zeros(b)]
    x = rng.uniform(-1.0, 1.0, (case["batch"], case["n_in"])).astype(np.float32)
    # profiles in [-1, 1]: smooth waves whose phase follows the inputs
    s = np.linspace(0.0, 1.0, case["n_out"])
    t = np.sin(2.0 * np.pi * s[None, :] * (1.0 + x[:, :1]) + np.pi * x[:, -1:]).astype(np.float32)
    return np.concatenate(p).astype(np.float32), x, t


# ---------------------------------------------------------------------------------
# The same in 64 bits, in plain numpy and torch
# ---------------------------------------------------------------------------------
def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "setup"):
        desc, M = _describe(case, seed), case["M"]
        if any(W.n_free(dm) * M > 8000 and not _splits(desc, d) for d, dm in enumerate(desc["dims"])):
            return None
        U0 = _splitmix_factors(desc, M, seed & 0xFFFFFF)
        U = _sweeps(desc, U0, case["sweeps"])
        U = [u.T for u in U] if kind == "solve" else U
        return dict(rho=None, rho_full=None, change=None, factors=[np.ascontiguousarray(u) for u in U])
    if kind == "batch":
        out = []
        for i, (ns, M, transient) in enumerate(_batch_layout(case)):
            desc = _poisson(ns, M, [seed, i], transient)
            U = _sweeps(desc, _random_factors(desc, M, seed + i), case["sweeps"])
            out.append(np.concatenate([u.T.reshape(-1) for u in U]))
        return dict(changes=None, factors=out)
    if kind == "nonlinear":
        return dict(changes=None, factors=_plate_stages(case, seed))
    if kind == "grid":
        desc = _grid_description(case)
        start, count, step = _slices(case, desc)
        rows = []
        for dm, u, s, c, t in zip(desc["dims"], _random_factors(desc, case["M"], seed), start, count, step):
            full = np.zeros((dm["n"], case["M"]))
            full[_free(dm)] = u
            rows.append(torch.tensor(full[s:s + t * c:t], device=_device()))
        lead = rows[0]
        for r in rows[1:-1]:
            lead = (lead[:, None, :] * r[None, :, :]).reshape(-1, case["M"])
        return (lead @ rows[-1].T).reshape(count)
    if kind == "points":
        desc = _poisson([case["n"]] * case["D"], 1, 0)
        pts = np.random.default_rng(seed).uniform(0.0, 1.0, (case["count"], case["D"]))
        prod = np.ones((case["count"], case["M"]))
        for d, (dm, u) in enumerate(zip(desc["dims"], _random_factors(desc, case["M"], seed))):
            full = np.zeros((dm["n"] + 2 * dm["s"], case["M"]))   # s zero rows on either side
            full[dm["s"]:dm["s"] + dm["n"]][_free(dm)] = u
            h = (dm["hi"] - dm["lo"]) / (dm["n"] - 1)
            e = np.clip(((pts[:, d] - dm["lo"]) / h).astype(int), 0, dm["n"] - 2)
            N, _ = _shape(dm, e, (pts[:, d] - dm["lo"]) / h - e)
            prod *= sum(N[:, k, None] * full[e + k] for k in range(2 * dm["s"] + 2))
        return prod.sum(axis=1)
    return _mlp_exact(case, seed)


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _free(dm):
    return np.arange(1 if dm["dirichlet_lo"] else 0, dm["n"] - (1 if dm["dirichlet_hi"] else 0))


def _shape(dm, e, t):
    """Shape functions and their derivatives at local coordinate t of element e (arrays):
    [point][2s + 2] for the nodes e - s .. e + 1 + s.  N = sum over the element's two nodes
    of the linear hat times the node's patch interpolant (cubic-spline kernels of width a h
    and monomials up to order p over the nodes within s elements)."""
    n, s, a, p = dm["n"], dm["s"], dm["a"], dm["p"]
    h = (dm["hi"] - dm["lo"]) / (n - 1)

    def spline(z):
        return np.where(z <= 0.5, 2 / 3 - 4 * z ** 2 + 4 * z ** 3,
                        np.where(z <= 1, 4 / 3 - 4 * z + 4 * z ** 2 - 4 / 3 * z ** 3, 0.0))

    def dspline(z):
        return np.where(z <= 0.5, -8 * z + 12 * z ** 2, np.where(z <= 1, -4 + 8 * z - 4 * z ** 2, 0.0))

    e, t = np.asarray(e), np.asarray(t, dtype=float)
    N, B = np.zeros((len(e), 2 * s + 2)), np.zeros((len(e), 2 * s + 2))
    for c in (0, 1):
        node = e + c
        hat, dhat = (1 - t, -1.0) if c == 0 else (t, 1.0)
        lo, hi = np.minimum(node, s), np.minimum(n - 1 - node, s)
        for nl, nr in set(zip(lo.tolist(), hi.tolist())):
            at = np.nonzero((lo == nl) & (hi == nr))[0]
            off = np.arange(-nl, nr + 1.0)
            na = len(off)
            G = np.zeros((na + p + 1, na + p + 1))
            G[:na, :na] = spline(np.abs(off[:, None] - off[None, :]) / a)
            G[:na, na:] = off[:, None] ** np.arange(p + 1)
            G[na:, :na] = G[:na, na:].T
            x = t[at] - c   # the point relative to the patch's own node
            r = x[:, None] - off
            q = np.arange(p + 1)
            row = np.concatenate([spline(np.abs(r) / a), x[:, None] ** q], axis=1)
            drow = np.concatenate([dspline(np.abs(r) / a) * np.sign(r) / a,
                                   q * x[:, None] ** np.maximum(q - 1, 0)], axis=1)
            Wv = np.linalg.solve(G, row.T)[:na].T
            dWv = np.linalg.solve(G, drow.T)[:na].T
            k = (off.astype(int) + c + s)
            N[at[:, None], k] += hat[at, None] * Wv
            B[at[:, None], k] += dhat * Wv + hat[at, None] * dWv
    return N, B / h


@functools.lru_cache(maxsize=64)
def _tables(key):
    dm = dict(key)
    n, s, nq = dm["n"], dm["s"], dm["n_quad"]
    h = (dm["hi"] - dm["lo"]) / (n - 1)
    g, w = np.polynomial.legendre.leggauss(nq)
    e = np.repeat(np.arange(n - 1), nq)
    t = np.tile(0.5 * (g + 1), n - 1)
    N, B = _shape(dm, e, t)
    return e, dm["lo"] + (e + t) * h, np.tile(0.5 * w * h, n - 1), N, B


def _key(dm):
    return tuple(sorted((k, tuple(v) if isinstance(v, (list, tuple)) else v) for k, v in dm.items()))


def _operator(dm, name, weight=None):
    """Dense 1D matrix over all nodes; `weight`: nodal values of a weight field (K, M, G)."""
    e, x, w, N, B = _tables(_key(dm))
    n, s = dm["n"], dm["s"]
    if name in ("Blo", "Bhi"):
        A = np.zeros((n, n))
        A[(0, 0) if name == "Blo" else (n - 1, n - 1)] = 1.0
        return A
    L, R = (B, B) if name == "K" else (N, N)
    if name == "G":
        R = B
    if name == "W":
        w = w * sum(c * x ** j for j, c in enumerate(dm["weight_poly"]))
    if weight is not None:
        pad = np.concatenate([np.zeros(s), weight, np.zeros(s)])
        vals = pad[e[:, None] + np.arange(2 * s + 2)]
        field, slope = (N * vals).sum(1), (B * vals).sum(1)
        R = slope[:, None] * N + field[:, None] * B if name == "G" else field[:, None] * R
    A = np.zeros((n + 2 * s, n + 2 * s))
    idx = e[:, None] + np.arange(2 * s + 2)
    np.add.at(A, (idx[:, :, None], idx[:, None, :]), w[:, None, None] * L[:, :, None] * R[:, None, :])
    return A[s:n + s, s:n + s]


def _source_vector(dm, kind, par):
    if kind == "nodal":
        return (_mass(_key(dm)) @ np.asarray(par, dtype=float))[_free(dm)]
    e, x, w, N, _ = _tables(_key(dm))
    g = {"const": lambda: np.full_like(x, par[0]), "sin": lambda: np.sin(par[0] * x + par[1]),
         "gauss": lambda: np.exp(-(x - par[0]) ** 2 / (2 * par[1] ** 2)),
         "poly": lambda: sum(c * x ** j for j, c in enumerate(par))}[kind]()
    q = np.zeros(dm["n"] + 2 * dm["s"])
    np.add.at(q, e[:, None] + np.arange(2 * dm["s"] + 2), N * (w * g)[:, None])
    return q[dm["s"]:dm["s"] + dm["n"]][_free(dm)]


@functools.lru_cache(maxsize=16)
def _mass(key):
    return _operator(dict(key), "M")


def _splits(desc, d):
    """Two operators of which one is a mass matrix: the reduced system decouples."""
    ops = {t[1][d] for t in desc["terms"]}
    return len(ops) <= 2 and bool(ops & {"M", "W"}) and ops <= {"K", "M", "W", "G"}


def _sweeps(desc, U, count, weights=None):
    """`count` sweeps of the subspace iteration; weights[d][name]: weighted operators."""
    dev = _device()
    dims, terms, D = desc["dims"], desc["terms"], len(desc["dims"])

    def t(x):
        return torch.tensor(np.ascontiguousarray(x), dtype=torch.float64, device=dev)

    ops = []
    for d, dm in enumerate(dims):
        f = _free(dm)
        names = dict.fromkeys(term[1][d] for term in terms)
        ops.append({k: t((weights[d][k] if k.startswith("w") else _operator(dm, k))[np.ix_(f, f)]) for k in names})
    Q = []
    for d, dm in enumerate(dims):
        seen = {}
        rows = []
        for _, facs in desc["sources"]:
            key = (facs[d][0], np.asarray(facs[d][1]).tobytes())
            if key not in seen:
                seen[key] = _source_vector(dm, *facs[d])
            rows.append(seen[key])
        Q.append(t(np.stack(rows)))
    beta = t(np.array([b for b, _ in desc["sources"]]))
    U = [t(u) for u in U]
    M = U[0].shape[1]
    for _ in range(count):
        for d in range(D):
            gram = [{k: U[e].T @ A @ U[e] for k, A in ops[e].items()} for e in range(D)]
            proj = [Q[e] @ U[e] for e in range(D)]
            C = {k: torch.zeros(M, M, dtype=torch.float64, device=dev) for k in ops[d]}
            for alpha, names in terms:
                c = torch.full((M, M), float(alpha), dtype=torch.float64, device=dev)
                for e in range(D):
                    if e != d:
                        c = c * gram[e][names[e]]
                C[names[d]] += c
            c = beta[:, None].repeat(1, M)
            for e in range(D):
                if e != d:
                    c = c * proj[e]
            X = _reduced(ops[d], C, Q[d].T @ c)
            if d < D - 1:
                big = X.abs().argmax(dim=0)
                X = X / (X.norm(dim=0) * torch.sign(X[big, torch.arange(M, device=dev)]))
            U[d] = X
    return [u.cpu().numpy() for u in U]


def _reduced(ops, C, F):
    """X with sum_o Op_o X C_o^T = F."""
    names = list(ops)
    n, M = F.shape
    mass = next((k for k in names if k in ("M", "W")), None)
    other = [k for k in names if k != mass]
    if len(names) <= 2 and mass and all(k in ("K", "M", "W") for k in other):
        L = torch.linalg.cholesky(ops[mass])
        if not other:
            return torch.linalg.solve(C[mass], torch.cholesky_solve(F, L).T).T
        S = torch.linalg.solve_triangular(L, ops[other[0]], upper=False)
        S = torch.linalg.solve_triangular(L, S.T, upper=False)
        mu, Z = torch.linalg.eigh(0.5 * (S + S.T))
        Phi = torch.linalg.solve_triangular(L.T, Z, upper=True)
        T = mu[:, None, None] * C[other[0]] + C[mass]
        return Phi @ torch.linalg.solve(T, (Phi.T @ F)[:, :, None])[:, :, 0]
    if len(names) == 2 and mass and other == ["G"]:
        L = torch.linalg.cholesky(0.5 * (C["G"] + C["G"].T))
        S = torch.linalg.solve_triangular(L, C[mass], upper=False)
        S = torch.linalg.solve_triangular(L, S.T, upper=False)
        lam, V = torch.linalg.eigh(0.5 * (S + S.T))
        Wm = torch.linalg.solve_triangular(L.T, V, upper=True)
        R = F @ Wm
        Z = [torch.linalg.solve(ops["G"] + lam[j] * ops[mass], R[:, j]) for j in range(M)]
        return torch.stack(Z, dim=1) @ Wm.T
    A = sum(torch.kron(ops[k], C[k]) for k in names)
    return torch.linalg.solve(A, F.reshape(-1)).reshape(n, M)


def _splitmix_factors(desc, M, seed):
    """U(-1, 1) draws of SplitMix64 keyed on (seed, dim, mode, row)."""
    out = []
    for d, dm in enumerate(desc["dims"]):
        i, m = np.meshgrid(np.arange(W.n_free(dm), dtype=np.uint64), np.arange(M, dtype=np.uint64), indexing="ij")
        z = (np.uint64(seed << 40) | np.uint64(d << 32) | (m << np.uint64(20)) | i) + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
        out.append(2.0 * ((z >> np.uint64(11)).astype(np.float64) / 9007199254740992.0) - 1.0)
    return out


def _plate_stages(case, seed):
    desc, M = _plate(case, seed), case["M"]
    m_c, n_c, m_k, n_k = W.INCONEL_LAW
    D = len(desc["dims"])
    terms = [(n_c, ["M"] * (D - 1) + ["G"])]
    terms += [(n_k, ["K" if d == e else "M" for d in range(D - 1)] + ["M"]) for e in range(D - 1)]
    U = _sweeps(dict(desc, terms=terms), _random_factors(desc, M, seed), case["sweeps"])
    for _ in range(case["stages"] - 1):
        weights, more = [dict() for _ in range(D)], []
        for j in range(M):
            for d, dm in enumerate(desc["dims"]):
                v = np.zeros(dm["n"])
                v[_free(dm)] = U[d][:, j]
                for base in "KM" if d < D - 1 else "GM":
                    weights[d][f"w{base}{j}"] = _operator(dm, base, v)
            more.append((m_c, [f"wM{j}"] * (D - 1) + [f"wG{j}"]))
            more += [(m_k, [f"wK{j}" if d == e else f"wM{j}" for d in range(D - 1)] + [f"wM{j}"]) for e in range(D - 1)]
        U = _sweeps(dict(desc, terms=terms + more), U, case["sweeps"], weights)
    return U


def _mlp_exact(case, seed):
    p, x, t = _mlp_inputs(case, seed)
    dims = [case["n_in"]] + [case["hidden"]] * case["layers"] + [case["n_out"]]
    p = torch.tensor(p, dtype=torch.float64)
    x, t = torch.tensor(x, dtype=torch.float64), torch.tensor(t, dtype=torch.float64)

    def forward(p):
        at, y = 0, x
        for k, (a, b) in enumerate(zip(dims, dims[1:])):
            y = y @ p[at:at + a * b].reshape(b, a).T + p[at + a * b:at + a * b + b]
            at += a * b + b
            y = torch.tanh(y) if k < len(dims) - 2 else y
        return y

    if not case["steps"]:
        return forward(p)
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    for k in range(1, case["steps"] + 1):
        q = p.clone().requires_grad_(True)
        loss = ((forward(q) - t) ** 2).mean()
        (g,) = torch.autograd.grad(loss, q)
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = p - 1e-3 * (m / (1 - 0.9 ** k)) / ((v / (1 - 0.999 ** k)).sqrt() + 1e-8)
    return dict(loss=loss.detach(), params=p)
