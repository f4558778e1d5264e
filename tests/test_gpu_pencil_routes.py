"""The kept node-side decomposition of a dim is the same whichever call makes it: a batch's
set-up and a single solve give the same bits, over the ranges of the tridiagonalisation's kernels
(a cluster's distributed shared memory, the whole chip's, one cluster on global memory)."""
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


@pytest.mark.parametrize("n", [300, 451, 600, 658, 659, 900, 1840])
def test_batch_and_single_set_up_agree(T, n):
    dims = [W.dim(n), W.dim(9)]
    rng = np.random.default_rng(n)
    sources = [(1.0, [("nodal", rng.uniform(-1, 1, dm["n"])) for dm in dims]) for _ in range(4)]
    desc = dict(name="pencil", dims=dims, terms=[(1.0, ["K", "M"]), (1.0, ["M", "K"])], sources=sources)
    U0 = W.random_factors(desc, 3, seed=n)

    def problem():
        stream = torch.cuda.Stream()
        P = T.Problem(desc, stream=T.ctypes.c_void_p(stream.cuda_stream))
        U = P.factors(3)
        U.set(U0)
        return P, U, stream

    fresh, member, other = problem(), problem(), problem()
    T.Batch([member[0], other[0]], [member[1], other[1]], solver=T.SOLVER_FASTDIAG)
    outs = []
    for P, U, _ in (fresh, member):   # the same sweep; the member's decomposition is the batch's
        P.sweep(U, 1, solver=T.SOLVER_FASTDIAG)
        outs.append(U.get())
    for a, b in zip(*outs):
        assert np.array_equal(a, b)
