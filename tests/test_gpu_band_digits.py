"""FP64 band factors and band solves by exact digit products, at their edges.

Matrices of less than one tile, of a few rows more than a tile, of wide bands
(every tile row coupled), graded ones (a permeability contrast of 1e7, clamped
rows of unit diagonal beside stiff ones) and coarse matrices whose size is no
multiple of the eight columns of a solve or of the 32 rows of a tile.

Tolerances.  Factor: |A - L L^T|_ij <= c sqrt(a_ii a_jj) is the form of the
backward error of a Cholesky factorisation; the digits and the FP64 storage of
L give c of a few 2^-53, the explicit inverses of the 32 x 32 diagonal blocks
(condition numbers up to about 1e4 here) 1e4 2^-53 = 1.1e-12.  Eigenvalues of
the shift-invert operator (both sweeps, many applications) 1e-7 relative, as
elsewhere.  Coarse correction: the GPU's own basis and A_H, solved densely;
condition numbers of A_H up to 1e5 allow 1e-9.
"""
import numpy as np
import pytest
import scipy.linalg as sla

from workloads.darcy import make_darcy
from workloads.laminate import make_block

from gpu_common import rel, require_gpu

pytestmark = pytest.mark.gpu

ANG = [0.0, 45.0, -45.0, 90.0]
PROBLEMS = {
    "under_a_tile": lambda: make_darcy(4, 2, 1, seed=1, partition=(2, 1, 1, 1)),
    "tile_and_a_bit": lambda: make_block(6, 1, 1, ANG[:1], partition=(2, 1, 1, 1)),
    "wide_band": lambda: make_block(7, 5, 4, ANG, partition=(2, 1, 1, 1)),
    "long_and_narrow": lambda: make_block(26, 2, 2, ANG[:2], partition=(2, 1, 1, 1)),
    "graded": lambda: make_darcy(12, 10, 9, seed=3, partition=(2, 1, 1, 1)),
    "resin": lambda: make_block(12, 9, 7, ANG, resin_between=True, partition=(2, 2, 1, 1)),
}


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


@pytest.fixture(params=sorted(PROBLEMS))
def solver(request, pkg):
    p = PROBLEMS[request.param]()
    p["modes"] = dict(fixed_modes=3, threshold=0.0, max_modes=20, shift=-0.01)
    s = pkg.GeneoSolver()
    s.assemble(p)
    s.setup(p, pkg.GENEO_FP64)
    yield s, p
    s.close()


def _lower(F):
    """L from the tile storage: the 32 x 32 diagonal blocks hold the inverses."""
    L = np.tril(F)
    for r in range(0, F.shape[0], 32):
        b = slice(r, min(F.shape[0], r + 32))
        L[b, b] = np.linalg.inv(np.tril(F[b, b]))
    return L


@pytest.mark.parametrize("kind", [3, 4])
def test_factor_backward_error(solver, kind):
    s, p = solver
    for j in range(s.part.px * s.part.py * s.part.pz):
        A, _ = s.local_matrix(j, kind - 3)
        L = _lower(s.local_matrix(j, kind)[0])
        d = np.sqrt(np.diag(A))
        assert np.max(np.abs(A - L @ L.T) / np.outer(d, d)) <= 1.1e-12, j


def test_eigenvalues_match_dense(solver):
    s, p = solver
    modes, lam, _ = s.coarse_info()
    sigma = p["modes"]["shift"]
    for j, m in enumerate(modes):
        S, _ = s.local_matrix(j, 1)
        B, _ = s.local_matrix(j, 2)
        mu = sla.eigh(B, S, eigvals_only=True)[::-1][:m]
        got = 1.0 / (lam[j, :m] - sigma)
        assert np.all(np.abs(got - mu) <= 1e-7 * mu), j


def test_coarse_correction_matches_dense(solver, pkg):
    s, p = solver
    Phi, AH = s.coarse()
    r = np.random.default_rng(0).normal(size=s.ndof)
    two = s.apply_preconditioner(r)
    s.setup(p, pkg.GENEO_FP64, pkg.GENEO_AS, pkg.GENEO_COARSE_NONE)
    one = s.apply_preconditioner(r)
    ref = Phi @ sla.solve(AH, Phi.T @ r, assume_a="pos")
    assert np.linalg.norm((two - one) - ref) <= 1e-9 * max(np.linalg.norm(ref), np.linalg.norm(two))
