"""Reduced solves at the edges of their kernels against the FP64 oracle: the mode-side banded
solves (every half-bandwidth, fewer nodes than the band, one to many systems, source counts
around the sixteen terms of a batch) and the node-side solves beyond 32 modes (one above the
limit, two and three row slots per lane)."""
import numpy as np
import pytest

from oracle import taps_oracle as O
from paper_2503_13933_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2503_13933_gb300 import build, taps
    import os
    if not os.path.exists(taps.LIB_PATH):
        build.build()
    taps.lib()
    return taps


def _nodal(dims, terms, count, seed):
    rng = np.random.default_rng(seed)
    sources = [(1.0, [("nodal", rng.uniform(-1, 1, dm["n"])) for dm in dims]) for _ in range(count)]
    return dict(name="nodal", dims=dims, terms=terms, sources=sources)


def _check(T, desc, M, seed, solver):
    U0 = W.random_factors(desc, M, seed=seed)
    P = T.Problem(desc)
    U = P.factors(M)
    U.set(U0)
    P.sweep(U, 1, solver=solver)
    Uo, _ = O.sweep(O.problem_from_description(desc), [u.copy() for u in U0])
    a, b = O.cp_full(U.get()), O.cp_full(Uo)
    # reduced systems of condition up to ~1e5: 1e5 eps and a factor for the dims
    assert np.linalg.norm(a - b) <= 1e-10 * np.linalg.norm(b)
    return P.profile()


@pytest.mark.parametrize("n_t,s,M,Rf", [(4, 2, 3, 5), (5, 2, 1, 1), (6, 2, 4, 15), (9, 1, 5, 16), (17, 2, 7, 17),
                                        (34, 2, 12, 33), (21, 1, 20, 48), (40, 2, 33, 40)])
def test_mode_side_time_solve(T, n_t, s, M, Rf):
    dims = [W.dim(14), W.dim(12), W.dim(n_t, s=s, p=min(s, 2), kind=W.TIME, dirichlet_lo=True, dirichlet_hi=False)]
    terms = [(1.0, ["M", "M", "G"]), (1.0, ["K", "M", "M"]), (1.0, ["M", "K", "M"])]
    prof = _check(T, _nodal(dims, terms, max(Rf, 1), n_t), M, M, T.SOLVER_FASTDIAG)
    assert prof["modediag"]["launches"] > 0


@pytest.mark.parametrize("M", [33, 64, 65, 97])
def test_node_side_beyond_32_modes(T, M):
    dims = [W.dim(18), W.dim(16), W.dim(15)]
    terms = [(1.0, ["K" if d == e else "M" for d in range(3)]) for e in range(3)]
    prof = _check(T, _nodal(dims, terms, M + 2, M), M, M, T.SOLVER_FASTDIAG)
    assert prof["fastdiag"]["launches"] > 0
