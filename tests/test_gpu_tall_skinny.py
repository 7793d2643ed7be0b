"""The block Lanczos products V^T W and V H by exact digits, at their edges.

Basis sizes of 80, 96 and 128 columns (the three widths the kernels distinguish,
met one after the other as the basis grows by eight), 3 and 24 modes (Gram
matrices of one and of several blocks), subdomains of fewer rows than a tile and
of a few more than a multiple of one, and a permeability contrast of 1e7, where
the columns of W differ in scale.

Tolerance.  With a Ritz residual of 1e-10 an eigenvalue mu of the shift-invert
operator is off by at most 1e-10 mu; loss of orthogonality in the basis (FP64
level after the second pass) and the products add a few 2^-53 n^(1/2) each, so
1e-9 relative leaves them a factor of ten.
"""
import numpy as np
import pytest
import scipy.linalg as sla

from workloads.darcy import make_darcy
from workloads.laminate import make_block

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

PROBLEMS = {
    "under_a_tile": lambda: make_darcy(4, 2, 1, seed=1, partition=(2, 1, 1, 1)),
    "ragged": lambda: make_block(9, 5, 4, [0.0, 45.0, -45.0, 90.0], partition=(2, 1, 1, 1)),
    "graded": lambda: make_darcy(12, 10, 9, seed=3, partition=(2, 1, 1, 1)),
}


@pytest.mark.parametrize("modes", [3, 24])
@pytest.mark.parametrize("steps", [10, 12, 16])
@pytest.mark.parametrize("name", sorted(PROBLEMS))
def test_eigenvalues(monkeypatch, name, steps, modes):
    pkg = require_gpu()
    monkeypatch.setenv("GENEO_LANCZOS_STEPS", str(steps))
    monkeypatch.setenv("GENEO_EIG_TOL", "1e-10")
    p = PROBLEMS[name]()
    p["modes"] = dict(fixed_modes=modes if name != "under_a_tile" else 3, threshold=0.0,
                      max_modes=24, shift=-0.01)
    s = pkg.GeneoSolver()
    s.assemble(p)
    s.setup(p, pkg.GENEO_FP64)
    counts, lam, _ = s.coarse_info()
    for j, m in enumerate(counts):
        S, _ = s.local_matrix(j, 1)
        B, _ = s.local_matrix(j, 2)
        mu = sla.eigh(B, S, eigvals_only=True)[::-1][:m]
        got = 1.0 / (lam[j, :m] - p["modes"]["shift"])
        assert np.all(np.abs(got - mu) <= 1e-9 * mu), j
    s.close()


def test_widest_mode_cap(monkeypatch):
    """A cap of 32 modes keeps 33 pairs: Gram matrices wider than a tile.

    The pairs at the cap lie in a dense part of the spectrum and are not all
    converged when the cycles end, so each Ritz value is held to the bound of a
    symmetric operator: an eigenvalue lies within its residual, which the
    statistics give relative to the value.
    """
    pkg = require_gpu()
    monkeypatch.setenv("GENEO_EIG_TOL", "1e-10")
    p = PROBLEMS["graded"]()
    p["modes"] = dict(fixed_modes=0, threshold=1e9, max_modes=32, shift=-0.01)
    s = pkg.GeneoSolver()
    s.assemble(p)
    s.setup(p, pkg.GENEO_FP64)
    counts, lam, _ = s.coarse_info()
    assert np.all(counts == 32)
    u, st = s.solve(tol=1e-8, max_it=500)
    for j, m in enumerate(counts):
        S, _ = s.local_matrix(j, 1)
        B, _ = s.local_matrix(j, 2)
        mu = sla.eigh(B, S, eigvals_only=True)
        got = 1.0 / (lam[j, :m] - p["modes"]["shift"])
        near = np.min(np.abs(got[:, None] - mu[None, :]), axis=1)
        assert np.all(near <= (1e-9 + st["eig_max_residual"]) * got), j
    Phi, AH = s.coarse()
    assert np.all(np.isfinite(Phi)) and np.all(np.linalg.eigvalsh(AH) > 0)
    assert st["rel_res_true"] <= 2e-6        # 2 tol, a factor of 100 for the contrast
    s.close()
