"""FP64 grid reconstruction at the edges of its 64 x 128 tiles, of their groups of 16 and of its
32-mode chunks, and FP32 at the same sizes, against the oracle's reconstruction at the nodes."""
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


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("counts,M", [((1, 1, 17), 1), ((3, 21, 127), 31), ((1, 64, 128), 32), ((5, 13, 129), 33),
                                      ((2, 33, 144), 65), ((7, 30, 12), 20)])
def test_grid_tile_edges(T, counts, M, dtype):
    dims = [W.dim(max(c + 3, 6)) for c in counts]
    desc = dict(name="grid", dims=dims, terms=[(1.0, ["M"] * 3)],
                sources=[(1.0, [("nodal", np.ones(dm["n"])) for dm in dims])])
    U0 = W.random_factors(desc, M, seed=M)
    P = T.Problem(desc)
    U = P.factors(M)
    U.set(U0)
    out = torch.full((int(np.prod(counts)),), float("nan"), dtype=torch.float64 if dtype == "f64" else torch.float32,
                     device="cuda")
    P.eval_grid(U, [1, 0, 2], list(counts), [1, 1, 1], out, dtype=T.FP64 if dtype == "f64" else T.FP32)
    torch.cuda.synchronize()
    ref = O.eval_grid(O.problem_from_description(desc), U0, [range(a, a + c) for a, c in zip([1, 0, 2], counts)])
    # the factors' entries are at most 1, so the M products and their partial sums are at most M:
    # M + 3 roundings (three of them of the factors and products) of half a unit each
    unit = 2.0 ** -53 if dtype == "f64" else 2.0 ** -24
    tol = (M + 3) * M * unit
    assert np.max(np.abs(out.double().cpu().numpy().reshape(ref.shape) - ref)) <= tol
