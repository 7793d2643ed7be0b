"""Subdomains of more than 65,536 unknowns: the products V^T W and W^T W of the
eigensolver add more 32-row tiles per chunk than their 32-bit sums hold, and turn
them into FP64 in between.

Eigenvalues against the oracle's (ARPACK on sparse factors of the same pencil),
1e-7 relative as elsewhere; a sum that overflowed would be wrong in the first digit.
"""
import numpy as np
import pytest

from oracle import decomp, geneo
from workloads.darcy import make_darcy

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


def test_eigenvalues_of_long_bars(monkeypatch):
    pkg = require_gpu()
    monkeypatch.setenv("GENEO_EIG_TOL", "1e-10")
    p = make_darcy(4, 4, 5260, partition=(1, 1, 2, 1),
                   modes=dict(fixed_modes=3, threshold=0.0, max_modes=20, shift=-0.01))
    rng = np.random.default_rng(2)
    p["perm"] = rng.uniform(0.5, 2.0, p["perm"].shape)
    subs = decomp.partition(p)
    assert min(s.neu_dofs.size for s in subs) > 65536
    s = pkg.GeneoSolver()
    s.assemble(p)
    s.setup(p, pkg.GENEO_FP64)
    counts, lam, _ = s.coarse_info()
    A, O = geneo.local_matrices(p, subs[0])
    X = np.asarray(subs[0].X)
    B = O.multiply(X[:, None]).multiply(X[None, :]).tocsr()
    ref, _ = geneo.eigenpairs(A, B, 4, p["modes"]["shift"])
    assert counts[0] == 3
    mu, got = (1.0 / (np.asarray(v)[:3] - p["modes"]["shift"]) for v in (ref, lam[0]))
    assert np.all(np.abs(got - mu) <= 1e-7 * mu)
    s.close()
