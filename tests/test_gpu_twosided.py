"""Block elimination from both ends against the FP64 oracle's banded solver, at the sizes
where its pieces change: no, one and two eliminated nodes beside the middle, every band
half-width, one and several columns per CTA, one and two row slots per lane (M = 32, 33),
the largest M of the route at s = 2 (37); beyond it and for s > 2 the one-ended elimination."""
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


def _transient(n, s, M, seed):
    """A transient problem (its time dim's reduced matrix is nonsymmetric) with M + 2 random
    separable nodal sources: right-hand sides of rank M, well conditioned reduced systems."""
    rng = np.random.default_rng(seed)
    p = min(s, 2)
    dims = [W.dim(n, s=s, p=p), W.dim(16, s=2),
            W.dim(n + 1, s=s, p=p, kind=W.TIME, dirichlet_lo=True, dirichlet_hi=False)]
    terms = [(1.0, ["M", "M", "G"]), (1.0, ["K", "M", "M"]), (1.0, ["M", "K", "M"])]
    sources = [(1.0, [("nodal", rng.uniform(-1, 1, dm["n"])) for dm in dims]) for _ in range(M + 2)]
    return dict(name="transient", dims=dims, terms=terms, sources=sources)


# free nodes of the first dim n - 2, of the time dim n; hb = 2 s + 1
@pytest.mark.parametrize("n,s,M", [(4, 2, 3), (7, 2, 5), (8, 2, 1), (9, 2, 4), (12, 2, 7), (15, 1, 6), (14, 3, 5),
                                   (16, 4, 6), (33, 2, 10), (40, 2, 17), (24, 2, 32), (24, 2, 33), (24, 2, 37),
                                   (24, 2, 38), (26, 1, 40)])
def test_block_elimination_matches_oracle(T, n, s, M):
    desc = _transient(n, s, M, seed=n + M)
    U0 = W.random_factors(desc, M, seed=M)
    P = T.Problem(desc)
    U = P.factors(M)
    U.set(U0)
    P.sweep(U, 1)   # the default solver
    Uo, _ = O.sweep(O.problem_from_description(desc), [u.copy() for u in U0])
    a, b = O.cp_full(U.get()), O.cp_full(Uo)
    # condition numbers of the reduced systems up to ~1e5 at these sizes: 1e5 eps with a
    # factor for the sum over the dims
    assert np.linalg.norm(a - b) <= 1e-10 * np.linalg.norm(b)
    assert P.profile()["block_lu"]["launches"] == 3
