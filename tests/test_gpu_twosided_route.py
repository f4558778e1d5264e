"""Which elimination a block solve takes, from the launch counts: one kernel and a back
substitution of its own from one end; from both ends the middle's kernel, after the two ends'
wherever nodes are left beside the middle (more than hb = 2 s + 1)."""
import numpy as np
import pytest

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


# free nodes n - 2; the first dim's order varies, the second's is s = 2 (14 free nodes)
@pytest.mark.parametrize("n,s,M,one_ended,with_ends", [
    (4, 2, 3, 0, 1), (7, 2, 5, 0, 1), (8, 2, 5, 0, 2), (5, 1, 4, 0, 1), (6, 1, 4, 0, 2), (24, 2, 32, 0, 2),
    (24, 2, 33, 0, 2), (24, 2, 37, 0, 2), (24, 2, 38, 2, 0), (26, 1, 40, 1, 1), (14, 3, 5, 1, 1), (16, 4, 6, 1, 1)])
def test_route_of_block_solves(T, n, s, M, one_ended, with_ends):
    rng = np.random.default_rng(M)
    dims = [W.dim(n, s=s, p=min(s, 2)), W.dim(16)]
    sources = [(1.0, [("nodal", rng.uniform(-1, 1, dm["n"])) for dm in dims]) for _ in range(M + 2)]
    desc = dict(name="route", dims=dims, terms=[(1.0, ["K", "M"]), (1.0, ["M", "K"])], sources=sources)
    P = T.Problem(desc)
    U = P.factors(M)
    U.set(W.random_factors(desc, M, seed=M))
    P.sweep(U, 1)   # the one-ended elimination's trials, which are not counted
    P.profile_reset(events=False)
    P.sweep(U, 1)
    count = {k: v["launches"] for k, v in P.profile().items()}
    assert count["block_lu"] == 2
    assert count["backsub"] == one_ended
    assert count["block_ends"] == with_ends
