"""Point evaluation through per-element polynomials against the FP64 oracle's evaluation
(Eq. 13), with the kernel that forms the shape functions at every point as the second
witness where the route excludes the polynomials."""
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


def _desc(D, n, s, p, a, n_quad):
    dims = [W.dim(n + 3 * d, -0.3, 1.1, s=s, p=p, a=a, n_quad=n_quad, dirichlet_lo=d % 2 == 0) for d in range(D)]
    terms = [(1.0, ["K" if d == e else "M" for d in range(D)]) for e in range(D)]
    return dict(name="points", dims=dims, terms=terms, sources=[(1.0, [("const", (1.0,))] * D)])


# odd and even mode counts around a pass (8 modes) of the kernel, every number of dims, the
# reproducing orders, the fewest Gauss points of the route (5) and fewer; dilations whose
# breakpoints lie on nodes, beyond the patch, and inside an element (3: the other kernel)
@pytest.mark.parametrize("D,n,s,p,a,nq,M,count", [
    (1, 9, 2, 2, 20.0, 6, 1, 5), (2, 12, 2, 2, 20.0, 6, 2, 129), (3, 20, 1, 1, 20.0, 6, 7, 1000),
    (4, 15, 3, 3, 20.0, 6, 8, 300), (5, 10, 4, 2, 20.0, 12, 9, 64), (6, 8, 2, 2, 20.0, 5, 16, 33),
    (7, 7, 2, 1, 20.0, 6, 17, 40), (8, 7, 2, 2, 20.0, 6, 33, 50), (3, 14, 2, 2, 4.0, 6, 5, 200),
    (3, 14, 2, 2, 3.0, 6, 5, 200), (2, 14, 2, 2, 20.0, 4, 5, 200)])
def test_points_match_oracle(T, D, n, s, p, a, nq, M, count):
    desc = _desc(D, n, s, p, a, nq)
    rng = np.random.default_rng(D * 100 + M)
    U0 = [rng.uniform(-1, 1, (W.n_free(dm), M)) for dm in desc["dims"]]
    pts = rng.uniform(-0.4, 1.2, (count, D))   # some outside: clamped
    # the ends, a node of every dim and just beside it
    x = np.array([np.linspace(dm["lo"], dm["hi"], dm["n"])[dm["n"] // 2] for dm in desc["dims"]])
    for k, row in enumerate([np.full(D, -0.3), np.full(D, 1.1), x, np.nextafter(x, 2.0)][:count]):
        pts[k] = row
    P = T.Problem(desc)
    U = P.factors(M + 3)
    U.set(U0)
    out = torch.full((count,), float("nan"), dtype=torch.float64, device="cuda")
    P.eval_points(U, torch.tensor(pts, device="cuda"), out)
    torch.cuda.synchronize()
    lo, hi = desc["dims"][0]["lo"], desc["dims"][0]["hi"]
    ref = O.eval_points(O.problem_from_description(desc), U0, np.clip(pts, lo, hi))
    # the patch moments lose up to ~1e5 eps (the oracle's and the tables' inverses alike) and
    # a product of D factors of order one carries D of those
    scale = np.max(np.abs(ref)) + 1e-300
    assert np.max(np.abs(out.cpu().numpy() - ref)) <= D * 3e-11 * scale
