"""Which kernels a point evaluation takes, from the nodes of its captured graph: two where the
per-element polynomials are formed and evaluated, one where the shape functions are formed at
every point."""
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


class Case:
    """A problem with factors and points on a stream of its own."""

    def __init__(self, T, D, n, M, count, a=20.0, n_quad=6):
        rng = np.random.default_rng(n + M)
        dims = [W.dim(n + d, a=a, n_quad=n_quad) for d in range(D)]
        terms = [(1.0, ["K" if d == e else "M" for d in range(D)]) for e in range(D)]
        self.desc = dict(name="points", dims=dims, terms=terms, sources=[(1.0, [("const", (1.0,))] * D)])
        self.U0 = [rng.uniform(-1, 1, (W.n_free(dm), M)) for dm in dims]
        self.pts = rng.uniform(0, 1, (count, D))
        self.stream = torch.cuda.Stream()
        self.handle = ctypes.c_void_p(self.stream.cuda_stream)
        self.P = T.Problem(self.desc, stream=self.handle)
        self.U = self.P.factors(M)
        self.U.set(self.U0)
        self.p = torch.tensor(self.pts, device="cuda")
        self.out = torch.full((count,), float("nan"), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()

    def evaluate(self, count=None):
        self.P.eval_points(self.U, self.p if count is None else self.p[:count], self.out)
        torch.cuda.synchronize()
        return self.out.cpu().numpy()

    def kernels(self, count=None, launch=False):
        """Nodes of the captured call; with launch, the graph is run once."""
        cu, graph, nodes = ctypes.CDLL("libcuda.so.1"), ctypes.c_void_p(), ctypes.c_size_t()
        assert cu.cuStreamBeginCapture_v2(self.handle, 2) == 0   # the relaxed mode
        try:
            self.P.eval_points(self.U, self.p if count is None else self.p[:count], self.out)
        finally:
            ended = cu.cuStreamEndCapture(self.handle, ctypes.byref(graph))
        assert ended == 0
        assert cu.cuGraphGetNodes(graph, None, ctypes.byref(nodes)) == 0
        if launch:
            ex = ctypes.c_void_p()
            assert cu.cuGraphInstantiateWithFlags(ctypes.byref(ex), graph, ctypes.c_ulonglong(0)) == 0
            assert cu.cuGraphLaunch(ex, self.handle) == 0
            torch.cuda.synchronize()
            cu.cuGraphExecDestroy(ex)
        cu.cuGraphDestroy(graph)
        return nodes.value


def _close(a, b, D):
    # the bound of the other point tests: 1e5 eps per dim for the patch moments
    return np.max(np.abs(a - b)) <= D * 3e-11 * np.max(np.abs(b))


def test_call_under_capture(T):
    """Without the polynomials' memory a captured call forms the shape functions, after an
    ordinary call it takes the polynomials; either graph gives the oracle's values."""
    c = Case(T, 3, 20, 5, 300)
    ref = O.eval_points(O.problem_from_description(c.desc), c.U0, c.pts)
    assert c.kernels(launch=True) == 1
    assert _close(c.out.cpu().numpy(), ref, 3)
    assert _close(c.evaluate(), ref, 3)
    c.out.fill_(float("nan"))
    torch.cuda.synchronize()
    assert c.kernels(launch=True) == 2
    assert _close(c.out.cpu().numpy(), ref, 3)


# the default dims; a dilation with a breakpoint inside an element; too few Gauss points
@pytest.mark.parametrize("a,n_quad,kernels", [(20.0, 6, 2), (4.0, 5, 2), (3.0, 6, 1), (20.0, 4, 1)])
def test_dims_of_the_polynomials(T, a, n_quad, kernels):
    c = Case(T, 2, 14, 5, 200, a=a, n_quad=n_quad)
    c.evaluate()
    assert c.kernels() == kernels


def test_few_points_of_long_dims(T):
    """Two dims of 2000 and 1999 elements, 40 modes: the polynomials cost 70 x 3999 x 40, a point
    without them 2 (300 + 2 x 40): 14733 points.  Short tables are always made."""
    c = Case(T, 2, 2000, 40, 14800)
    c.evaluate()
    limit = 70 * (1999 + 2000) * 40 // ((300 + 2 * 40) * 2)
    assert c.kernels(1) == 1
    assert c.kernels(limit) == 1
    assert c.kernels(limit + 1) == 2
    general = c.evaluate(limit)[:limit].copy()
    assert _close(c.evaluate(limit + 1)[:limit], general, 2)
    s = Case(T, 2, 60, 40, 1)
    s.evaluate()
    assert s.kernels() == 2
