"""The node-side decomposition's kernels for the largest dims against the FP64 oracle: inverse
iteration of one eigenvector to a CTA, the Cholesky factor of a band that leaves shared memory,
and inverse iteration on global arrays."""
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


# with 227 KB a CTA: one vector to a CTA from ~2820 nodes, none from ~4720; the factor of a band
# of s = 4 leaves shared memory at ~2890
@pytest.mark.parametrize("n,s", [(2880, 4), (2910, 4), (4750, 1)])
def test_sweep_of_long_dims(T, n, s):
    dims = [W.dim(n, s=s, p=min(s, 2)), W.dim(9)]
    rng = np.random.default_rng(n)
    sources = [(1.0, [("nodal", rng.uniform(-1, 1, dm["n"])) for dm in dims]) for _ in range(4)]
    desc = dict(name="pencil", dims=dims, terms=[(1.0, ["K", "M"]), (1.0, ["M", "K"])], sources=sources)
    U0 = W.random_factors(desc, 3, seed=n)
    P = T.Problem(desc)
    U = P.factors(3)
    U.set(U0)
    P.sweep(U, 1, solver=T.SOLVER_FASTDIAG)
    Uo, _ = O.sweep(O.problem_from_description(desc), [u.copy() for u in U0])
    a, b = O.cp_full(U.get()), O.cp_full(Uo)
    # a decomposition is backward stable: relative error eps times the ratio of the pencil's ends,
    # below 16 n^2 / pi^2, and ten for the other dim and the oracle's own solve
    tol = 10 * 2.2e-16 * 16 * n * n / np.pi ** 2
    assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b)
