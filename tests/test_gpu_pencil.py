"""The node-side decomposition over its kernels' ranges against the FP64 oracle: one sweep of a
two-dim problem whose first dim has every half-bandwidth, fewer nodes than the band, and node
counts on both sides of the limits at which the tridiagonalisation (cluster or whole chip),
the Cholesky factor and the inverse iteration (eight, four, two columns to a CTA) change."""
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


@pytest.mark.parametrize("n,s", [(5, 1), (6, 2), (8, 3), (10, 4), (35, 1), (130, 3), (257, 4), (449, 2), (450, 2),
                                 (451, 1), (828, 2), (829, 2), (1000, 1), (1540, 2), (1566, 1), (1900, 1)])
def test_sweep_over_pencil_sizes(T, n, s):
    dims = [W.dim(n, s=s, p=min(s, 2)), W.dim(9)]
    terms = [(1.0, ["K", "M"]), (1.0, ["M", "K"])]
    rng = np.random.default_rng(n)
    sources = [(1.0, [("nodal", rng.uniform(-1, 1, dm["n"])) for dm in dims]) for _ in range(4)]
    desc = dict(name="pencil", dims=dims, terms=terms, sources=sources)
    U0 = W.random_factors(desc, 3, seed=n)
    P = T.Problem(desc)
    U = P.factors(3)
    U.set(U0)
    P.sweep(U, 1, solver=T.SOLVER_FASTDIAG)
    Uo, _ = O.sweep(O.problem_from_description(desc), [u.copy() for u in U0])
    a, b = O.cp_full(U.get()), O.cp_full(Uo)
    # a decomposition is backward stable: relative error eps times the ratio of the pencil's ends,
    # below 16 n^2 / pi^2, and ten for the other dim and the oracle's own solve; 1e5 eps is the
    # reduced systems' floor in the other tests of this kind
    tol = max(1e-10, 10 * 2.2e-16 * 16 * n * n / np.pi ** 2)
    assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b)


def test_batch_set_up_over_pencil_sizes(T):
    """Decompositions side by side (a batch): cluster tridiagonalisations of more entries than a
    CTA has threads, in distributed shared memory and in global memory."""
    sizes = [300, 515, 560, 600, 644, 660, 700, 1000]
    Ps, Us, descs, U0s = [], [], [], []
    for n in sizes * 2:
        dims = [W.dim(n), W.dim(9)]
        rng = np.random.default_rng(n)
        sources = [(1.0, [("nodal", rng.uniform(-1, 1, dm["n"])) for dm in dims]) for _ in range(4)]
        desc = dict(name="pencil", dims=dims, terms=[(1.0, ["K", "M"]), (1.0, ["M", "K"])], sources=sources)
        U0 = W.random_factors(desc, 3, seed=n)
        stream = torch.cuda.Stream()
        P = T.Problem(desc, stream=T.ctypes.c_void_p(stream.cuda_stream))
        U = P.factors(3)
        U.set(U0)
        Ps.append(P), Us.append(U), descs.append((desc, stream)), U0s.append(U0)
    T.Batch(Ps, Us, solver=T.SOLVER_FASTDIAG).sweep(1)
    torch.cuda.synchronize()
    for n, (desc, _), U, U0 in zip(sizes, descs, Us, U0s):
        Uo, _ = O.sweep(O.problem_from_description(desc), [u.copy() for u in U0])
        a, b = O.cp_full(U.get()), O.cp_full(Uo)
        tol = max(1e-10, 10 * 2.2e-16 * 16 * n * n / np.pi ** 2)   # as above
        assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b), n
