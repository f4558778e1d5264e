"""Backward error of the reduced solves of the two-sided block elimination.

The reduced matrix is M_0 (x) G with G = U_1^T M_1 U_1 and U_1 chosen so that G = R^T R with R
Kahan's triangle: symmetric positive definite, of condition 1e14 to 1e15, and with a triangular
factor whose inverse is far larger than its norms show.  LU without pivoting leaves a residual
of some eps there whatever the condition; what multiplies by (part of) an inverse, as Gauss-Jordan
elimination does, leaves thousands of eps."""
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


def _kahan(M, theta):
    c, s = np.cos(theta), np.sin(theta)
    return s ** np.arange(M)[:, None] * (np.eye(M) - c * np.triu(np.ones((M, M)), 1))


def _lu_growth(G):
    """|| |L| |U| || / ||G|| of LU without pivoting."""
    L, U = np.eye(len(G)), G.copy()
    for p in range(len(G) - 1):
        L[p + 1:, p] = U[p + 1:, p] / U[p, p]
        U[p + 1:] -= np.outer(L[p + 1:, p], U[p])
        U[p + 1:, p] = 0.0
    return np.abs(np.abs(L) @ np.abs(U)).sum(1).max() / np.abs(G).sum(1).max()


# one block (the middle alone) and a band from both ends; one and two row slots per lane
@pytest.mark.parametrize("n,M,theta", [(3, 24, 0.9), (24, 24, 0.9), (3, 32, 1.1), (24, 32, 1.1), (3, 36, 1.1),
                                       (24, 36, 1.1)])
def test_reduced_solve_backward_error(T, n, M, theta):
    worst = 0.0
    for seed in range(4):
        rng = np.random.default_rng(seed)
        dims = [W.dim(n, s=1, p=1), W.dim(60)]
        desc = dict(name="kahan", dims=dims, terms=[(1.0, ["M", "M"])],
                    sources=[(1.0, [("nodal", np.ones(dm["n"])) for dm in dims])])
        M1 = O.problem_from_description(desc).ops[1][1]
        Q = np.linalg.qr(rng.standard_normal((len(M1), M)))[0]
        U1 = np.linalg.solve(np.linalg.cholesky(M1).T, Q @ _kahan(M, theta))
        v = np.zeros(60)
        v[1:-1] = U1 @ rng.uniform(-1, 1, M)   # a right-hand side G x with x of order one
        desc["sources"] = [(1.0, [("nodal", rng.uniform(-1, 1, n)), ("nodal", v)])]
        P = T.Problem(desc)
        U = P.factors(M)
        U.set([rng.uniform(-1, 1, (W.n_free(dims[0]), M)), U1])
        P.refresh_grams(U)
        gram, h, ops = P.grams(1, M)
        G = gram[ops.index(T.OP["M"])]
        band, nf, hb = P.op_band(0, "M"), P.n_free[0], P.dims[0].hb
        M0 = np.zeros((nf, nf))
        for i in range(nf):
            for k in range(2 * hb + 1):
                if 0 <= i + k - hb < nf:
                    M0[i, i + k - hb] = band[i, k]
        P.sweep(U, 1, normalize=False)   # the default solver; dim 0 is solved first, from these Grams
        X = U.get()[0]
        F = np.outer(P.source(0, 0), h[0])
        R = F - M0 @ X @ G.T
        scale = np.abs(np.kron(M0, G)).sum(1).max() * np.abs(X).max() + np.abs(F).max()
        eta = np.abs(R).max() / scale
        # LU of a matrix and its two triangular solves: 3 M u || |L| |U| ||, for each of the
        # hb + 1 block rows that a row of the band passes through
        bound = 3 * M * 1.1e-16 * _lu_growth(G) * (min(hb, nf - 1) + 1)
        worst = max(worst, eta / bound)
        print(f"n {n} M {M} seed {seed}: backward error {eta:.1e}, bound {bound:.1e}, cond {np.linalg.cond(G):.0e}")
    assert worst <= 1.0
