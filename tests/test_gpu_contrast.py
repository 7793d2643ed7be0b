"""Set-ups with a permeability that jumps by 1e10 and 1e12 from cell to cell.

The eigensolver's factors, sweeps and products then meet rows and columns of very
different size.  Each Ritz value lies within its residual of an eigenvalue of the
dense pencil (the bound of a symmetric operator), and within 1e-9 for the rest
(loss of orthogonality and rounding, a few 2^-53 n^(1/2), with a factor of ten to
spare).  The solution against a dense one: the iteration's true residual, relative
to the load, carried by the condition number of the diagonally scaled matrix.
"""
import numpy as np
import pytest
import scipy.linalg as sla

from oracle import darcy
from workloads.darcy import make_darcy

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("power", [10, 12])
@pytest.mark.parametrize("prec", [0, 1])
def test_random_two_level_permeability(monkeypatch, power, prec):
    pkg = require_gpu()
    monkeypatch.setenv("GENEO_EIG_TOL", "1e-10")
    p = make_darcy(12, 9, 8, seed=1, partition=(2, 1, 1, 1))
    k = 10.0 ** (power * np.random.default_rng(power).integers(0, 2, p["nx"] * p["ny"] * p["nz"]))
    p["perm"] = np.stack([k, k, k], axis=1)
    p["modes"] = dict(fixed_modes=0, threshold=0.0, max_modes=20, shift=-0.01)
    s = pkg.GeneoSolver()
    s.assemble(p)
    s.setup(p, prec)
    counts, lam, _ = s.coarse_info()
    u, st = s.solve(tol=1e-8, max_it=2000)
    for j, m in enumerate(counts):
        S, _ = s.local_matrix(j, 1)
        B, _ = s.local_matrix(j, 2)
        d = 1.0 / np.sqrt(np.diag(S))
        mu = sla.eigh(d[:, None] * B * d, d[:, None] * S * d, eigvals_only=True)
        got = 1.0 / (lam[j, :m] - p["modes"]["shift"])
        near = np.min(np.abs(got[:, None] - mu[None, :]), axis=1)
        assert np.all(near <= (1e-9 + st["eig_max_residual"]) * got), j
    A, b = darcy.assemble_system(p)
    d = 1.0 / np.sqrt(A.diagonal())
    D = (A.toarray() * d) * d[:, None]
    w = np.linalg.eigvalsh(D)
    ref = d * np.linalg.solve(D, d * b)
    err = np.linalg.norm((u - ref) / d) / np.linalg.norm(ref / d)
    res = np.linalg.norm(d * (b - A @ u)) / w[0]
    assert err * np.linalg.norm(ref / d) <= 1.01 * res + 1e-9 * np.linalg.norm(ref / d)
    assert st["rel_res_true"] <= 1e-6
    s.close()
