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

from workloads.darcy import make_darcy

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


def _lower(F):
    """L from the tile storage: the 32 x 32 diagonal blocks hold the inverses."""
    L = np.tril(F).astype(np.longdouble)
    for r in range(0, F.shape[0], 32):
        D = np.tril(F[r:r + 32, r:r + 32]).astype(np.longdouble)
        X = np.zeros_like(D)
        for i in range(D.shape[0]):
            X[i, i] = 1 / D[i, i]
            X[i, :i] = -(D[i, :i] @ X[:i, :i]) * X[i, i]
        L[r:r + 32, r:r + 32] = X
    return L


@pytest.mark.parametrize("bits", [0, 6, 17, 24])
@pytest.mark.parametrize("n,hb", [(31, 3), (200, 40), (270, 100), (270, 270)])
def test_coefficients_that_vary_within_a_tile(ctx, n, hb, bits):
    """A = S M S with S_ii in {1, 2^bits} at random: a contrast of up to 3e14 from row to row.

    Cholesky is invariant under such a scaling, so the errors are M's.  Backward
    error relative to sqrt(a_ii a_jj): two subtractions and the rounding of L leave
    at most 8 u outside the diagonal blocks (of which L is taken as the exact inverse of what is
    stored); inside, 32 eliminations and the inverse 150 u.  L, and
    the solutions scaled back, equal those of M but for the pivots' reciprocals
    (a few u, carried by the condition number 3): 100 u of the largest in the row or column.
    """
    import paper_1901_05188_gb300 as pkg
    M = _matrix(n, hb)
    S = np.where(np.random.default_rng(bits).integers(0, 2, n) == 1, 2.0 ** bits, 1.0)
    A = S[:, None] * M * S[None, :]
    F0, F = np.zeros((n, n)), np.zeros((n, n))
    pkg.geneo_debug_band(ctx, M, hb, F0)
    pkg.geneo_debug_band(ctx, A, hb, F)
    L0, L = _lower(F0), _lower(F)
    d = np.sqrt(np.diag(A))
    E = np.abs(np.tril((A - L @ L.T) / np.outer(d, d)))
    tile = np.arange(n) // 32
    inside = tile[:, None] == tile[None, :]
    assert E[~inside].max(initial=0) <= 8 * U
    assert E[inside].max() <= 150 * U
    top = np.abs(L0).max(axis=1)[:, None]
    assert np.max(np.abs(L / S[:, None] - L0) / top) <= 100 * U
    b = np.random.default_rng(5).normal(size=(n, 9))
    # L x = S b and L^T x = b: the solutions of M, the second divided by S
    for mode, rhs, back in ((1, S[:, None] * b, 1.0), (2, b, S[:, None]), (3, S[:, None] * b, S[:, None])):
        x0, x = _solve(ctx, M, hb, b, mode), _solve(ctx, A, hb, rhs, mode) * back
        assert np.max(np.abs(x - x0)) <= 100 * U * np.abs(x0).max(), mode


@pytest.mark.parametrize("entry", [3.95, 8.1, 12.0, 1e3, 1e6, 1e200, np.inf, np.nan])
@pytest.mark.parametrize("at", [(40, 0), (33, 31), (95, 0), (95, 33)])
def test_indefinite_matrices_are_refused(ctx, at, entry):
    """3.9 on the diagonal and one larger entry beside it, in every launch that
    forms a tile: the tile below the diagonal and those further down."""
    import paper_1901_05188_gb300 as pkg
    A = 3.9 * np.eye(96)
    A[at] = A[at[::-1]] = 3.85
    F = np.zeros((96, 96))
    pkg.geneo_debug_band(ctx, A, 96, F)
    assert abs(F[at] * F[at[1], at[1]] - 3.85 / 3.9) <= 16 * U    # L_ij / L_jj, the inverse stored
    A[at] = A[at[::-1]] = entry
    with pytest.raises(pkg.GeneoError) as e:
        pkg.geneo_debug_band(ctx, A, 96, F)
    assert e.value.status == 4                                   # GENEO_ERR_NOT_SPD


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("coarse", ["GENEO_COARSE_NONE", "GENEO_COARSE_GENEO"])
def test_a_negative_permeability_is_refused(prec, coarse):
    pkg = require_gpu()
    p = make_darcy(12, 6, 5, seed=2, partition=(2, 1, 1, 1))
    p["perm"] = p["perm"].copy()
    p["perm"][72:216] *= -1.0         # two layers: the nodes between them have negative diagonals
    s = pkg.GeneoSolver()
    s.assemble(p)
    with pytest.raises(pkg.GeneoError) as e:
        s.setup(p, prec, pkg.GENEO_AS, getattr(pkg, coarse))
    assert e.value.status == 4
    s.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("n,hb,ctas", [(270, 40, 1), (420, 192, 2), (90, 0, 1), (20, 3, 1)])
def test_a_right_hand_side_that_is_not_finite_stays_so(ctx, n, hb, ctas, bad):
    """As with dense tiles: from the tile of the bad row on (backward: up to it; an
    uncoupled matrix: in it), in its column only."""
    A = _matrix(n, hb)
    rng = np.random.default_rng(3)
    b = rng.normal(size=(n, 11))
    i, c = n // 2, 9
    tile, I = np.arange(n) // 32, (n // 2) // 32
    worse = b.copy()
    worse[i, c] = bad
    for mode in (1, 2, 3):
        good, x = _solve(ctx, A, hb, b, mode, ctas), _solve(ctx, A, hb, worse, mode, ctas)
        other = np.arange(11) != c
        assert np.array_equal(good[:, other], x[:, other])
        hit = tile == I if hb == 0 else tile >= I if mode == 1 else tile <= I if mode == 2 else tile >= 0
        assert not np.any(np.isfinite(x[hit, c])), mode
        assert np.array_equal(x[~hit, c], good[~hit, c]), mode


@pytest.mark.parametrize("power", [-980, -960, -512, 512, 960])
@pytest.mark.parametrize("n,hb", [(31, 3), (200, 40), (270, 270)])
def test_small_and_large_matrices(ctx, n, hb, power):
    """2^power M: products of digits whose scales lie near the ends of the FP64 range.

    The factor and the solutions are M's times powers of two, but for the pivots'
    reciprocals (a few u, carried by the condition number 3): 100 u of the largest.
    """
    import paper_1901_05188_gb300 as pkg
    M, s = _matrix(n, hb), 2.0 ** (power // 2)
    F0, F = np.zeros((n, n)), np.zeros((n, n))
    pkg.geneo_debug_band(ctx, M, hb, F0)
    pkg.geneo_debug_band(ctx, M * s * s, hb, F)
    tile = np.arange(n) // 32
    F = np.where(tile[:, None] == tile[None, :], F * s, F / s)
    assert np.max(np.abs(F - F0)) <= 100 * U * np.abs(F0).max()
    b = np.random.default_rng(5).normal(size=(n, 9))
    for mode, back in ((1, s), (2, s), (3, s)):
        x0 = _solve(ctx, M, hb, b, mode)
        x = _solve(ctx, M * s * s, hb, b if mode < 3 else b * s, mode) * back
        assert np.max(np.abs(x - x0)) <= 100 * U * np.abs(x0).max(), mode


def test_more_tiles_than_one_sum_of_level_sums_holds(ctx):
    """A full matrix of 264 tile rows: with one CTA a warp adds up to 65 tiles of
    a row, one more than its 32-bit sums hold; with two CTAs 33.

    A = 2 I + V V^T with ||V V^T|| = 2 (condition number at most 2) has the inverse
    (I - V (2 I + V^T V)^-1 V^T) / 2; bound as above.
    """
    n = 264 * 32 - 5
    rng = np.random.default_rng(8)
    V = np.linalg.qr(rng.normal(size=(n, 4)))[0] * np.sqrt([2.0, 1.5, 1.0, 0.5])
    A = V @ V.T
    A[np.arange(n), np.arange(n)] += 2.0
    b = rng.normal(size=(n, 3))
    ref = 0.5 * (b - V @ np.linalg.solve(2.0 * np.eye(4) + V.T @ V, V.T @ b))
    one = _solve(ctx, A, n, b, 3, 1)
    assert np.linalg.norm(one - ref) <= 24 * n * U * np.linalg.norm(ref)
    assert np.max(np.abs(one - _solve(ctx, A, n, b, 3, 2))) <= 8 * U * np.abs(one).max()
