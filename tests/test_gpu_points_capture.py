"""Point evaluation and stream captures: a first evaluation on a factor set, which allocates its
polynomials' memory, leaves a capture of another stream in the global mode valid."""
import ctypes

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


def _problem(T):
    dims = [W.dim(20), W.dim(16), W.dim(12)]
    terms = [(1.0, ["K" if d == e else "M" for d in range(3)]) for e in range(3)]
    desc = dict(name="points", dims=dims, terms=terms, sources=[(1.0, [("const", (1.0,))] * 3)])
    stream = torch.cuda.Stream()
    P = T.Problem(desc, stream=ctypes.c_void_p(stream.cuda_stream))
    return desc, stream, P


def test_first_evaluation_beside_a_global_capture(T):
    M, count = 5, 700
    desc, stream, P = _problem(T)
    rng = np.random.default_rng(7)
    U0 = [rng.uniform(-1, 1, (W.n_free(dm), M)) for dm in desc["dims"]]
    pts = rng.uniform(0, 1, (count, 3))
    with torch.cuda.stream(stream):
        p = torch.tensor(pts, device="cuda")
        out = torch.full((count,), float("nan"), dtype=torch.float64, device="cuda")
    warm, U = P.factors(M), P.factors(M)
    warm.set(U0)
    U.set(U0)
    P.eval_points(warm, p, out)   # the kernels' code is loaded
    torch.cuda.synchronize()
    out.fill_(float("nan"))
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    other, graph = torch.cuda.Stream(), ctypes.c_void_p()
    other_h = ctypes.c_void_p(other.cuda_stream)
    assert cu.cuStreamBeginCapture_v2(other_h, 0) == 0   # the global mode
    try:
        P.eval_points(U, p, out)
    finally:
        ended = cu.cuStreamEndCapture(other_h, ctypes.byref(graph))
    if graph.value:
        cu.cuGraphDestroy(graph)
    assert ended == 0
    torch.cuda.synchronize()
    ref = O.eval_points(O.problem_from_description(desc), U0, pts)
    # the bound of the other point tests: 1e5 eps per dim for the patch moments
    assert np.max(np.abs(out.cpu().numpy() - ref)) <= 3 * 3e-11 * np.max(np.abs(ref))
