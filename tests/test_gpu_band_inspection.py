"""The FP64 band factorisation and band solves on given matrices.

M = 4 I + G with a symmetric random band G, ||G||_inf = 2, has condition number at
most 3.  Sizes: one row, a tile less and a tile more one row, a diagonal matrix,
half-bandwidths of 5 and 6 tiles (where the set-up's rule begins to use a second
CTA) and a full matrix, with column counts off the eight of a cluster.

Tolerances, u = 2^-53.  Solutions against dense ones: backward errors of both are
below n u, so 8 n u cond = 24 n u leaves a factor of four.  One and two CTAs add
the same integers, but for the bits dropped when sums of different scales are
aligned (below 2^-57 of the largest): they may turn the rounding of an entry, 1 u
in each sweep, which the condition number carries to 4 u; 8 u.
"""
import numpy as np
import pytest

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

U = 2.0 ** -53
SHAPES = [(1, 0), (31, 3), (33, 32), (200, 40), (90, 0), (420, 160), (420, 192), (270, 270)]


@pytest.fixture(scope="module")
def ctx():
    s = require_gpu().GeneoSolver()
    yield s.ctx
    s.close()


def _matrix(n, hb, seed=0):
    rng = np.random.default_rng(seed + 1000 * n + hb)
    G = np.tril(rng.normal(size=(n, n)))
    G[np.subtract.outer(np.arange(n), np.arange(n)) > hb] = 0.0
    G = G + np.tril(G, -1).T
    return 4.0 * np.eye(n) + G * (2.0 / np.abs(G).sum(axis=1).max())


def _solve(ctx, A, hb, b, mode=3, ctas=0):
    import paper_1901_05188_gb300 as pkg
    x = np.zeros_like(b)
    pkg.geneo_debug_band(ctx, A, hb, None, b, x, mode, ctas)
    return x


@pytest.mark.parametrize("n,hb", SHAPES)
@pytest.mark.parametrize("ncols", [1, 8, 13])
def test_solves_match_dense_with_one_and_two_ctas(ctx, n, hb, ncols):
    A = _matrix(n, hb)
    b = np.random.default_rng(ncols).normal(size=(n, ncols))
    L = np.linalg.cholesky(A)
    for mode, ref in ((1, np.linalg.solve(L, b)), (2, np.linalg.solve(L.T, b)), (3, np.linalg.solve(A, b))):
        one = _solve(ctx, A, hb, b, mode, 1)
        assert np.linalg.norm(one - ref) <= 24 * n * U * np.linalg.norm(ref), mode
        assert np.max(np.abs(one - _solve(ctx, A, hb, b, mode, 2))) <= 8 * U * np.abs(one).max(), mode
