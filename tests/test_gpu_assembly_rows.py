"""Row-wise assembly against the oracle at the sizes where its blocks end.

One-element axes (two-node rows of the pattern), node counts around a block of
32 (elasticity) or 128 (Darcy) nodes, graded axes with three distinct element
sizes, wrinkled plies of distinct moduli, Dirichlet values off zero scattered
over single components, and subdomains with and without overlap elements.
Entries: the oracle integrates with 2x2x2 Gauss points, exact for the closed
form used here, so both differ by rounding only: 1e-12 of the largest entry;
the load sums at most 81 products per row: 1e-12 of the largest.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import darcy, decomp, fem, geneo
from workloads.darcy import make_darcy
from workloads.laminate import make_block

from gpu_common import bsr_to_csr, require_gpu

pytestmark = pytest.mark.gpu

SIZES = [(1, 1, 2), (2, 1, 3), (7, 1, 4), (30, 1, 2), (31, 3, 2), (5, 7, 6)]


@pytest.fixture(scope="module")
def pkg():
    return require_gpu()


def _problem(physics, size, parts):
    nx, ny, nz = size
    rng = np.random.default_rng(nx + 10 * ny + 100 * nz)
    if physics == "darcy":
        p = make_darcy(nx, ny, nz, seed=nz, partition=(*parts, 1))
        p["perm"] = p["perm"] * rng.uniform(0.5, 2.0, p["perm"].shape)
    else:
        p = make_block(nx, ny, nz, [30.0, -70.0], partition=(*parts, 1), wrinkle=(20.0, 2.0))
        p["materials"][0] = (150e3, 12e3, 9e3, 5e3, 4e3, 3e3, 0.3, 0.25, 0.4)
    for k in "xyz":
        p[k] = np.concatenate([[0.0], np.cumsum(rng.uniform(0.3, 1.5, p["n" + k]))])
    nc = 1 if physics == "darcy" else 3
    n = nc * (nx + 1) * (ny + 1) * (nz + 1)
    dofs = np.unique(np.concatenate([p["dirichlet_dofs"], rng.integers(0, n, max(1, n // 20))]))
    p["dirichlet_dofs"] = dofs.astype(np.int32)
    p["dirichlet_values"] = rng.normal(size=dofs.size)
    return p, nc


@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("physics", ["elastic", "darcy"])
def test_rows_match_oracle(pkg, physics, size):
    p, nc = _problem(physics, size, (1, 1, 1))
    s = pkg.GeneoSolver()
    s.assemble(p)
    rp, col, val, b = s.system()
    Ao, bo = (darcy if nc == 1 else fem).assemble_system(p)
    cnt = np.full((p["nz"] + 1, p["ny"] + 1, p["nx"] + 1), 1)
    for ax, n in zip((2, 1, 0), (p["nx"], p["ny"], p["nz"])):
        w = np.full(n + 1, 3)
        w[0] = w[-1] = 2
        cnt = cnt * w.reshape([-1 if a == ax else 1 for a in range(3)])
    assert np.array_equal(np.diff(rp), cnt.reshape(-1)) and rp[0] == 0
    assert abs(bsr_to_csr(rp, col, val, s.nnode, nc) - Ao).max() <= 1e-12 * abs(Ao).max()
    assert np.abs(b - bo).max() <= 1e-12 * np.abs(bo).max()
    s.close()


@pytest.mark.parametrize("physics,size,parts", [("elastic", (7, 3, 6), (2, 1, 1)),
                                                ("elastic", (9, 8, 4), (3, 2, 1)),
                                                ("darcy", (14, 9, 5), (2, 2, 1)),
                                                ("darcy", (6, 5, 12), (1, 1, 3))])
def test_neumann_rows_match_oracle(pkg, physics, size, parts):
    p, nc = _problem(physics, size, parts)
    s = pkg.GeneoSolver()
    s.assemble(p)
    try:
        s.setup(p, pkg.GENEO_FP64)
    except pkg.GeneoError:
        pass          # the matrices are checked even if a later set-up step fails
    sigma = p["modes"]["shift"]
    for j, sd in enumerate(decomp.partition(p)):
        An, Ao = geneo.local_matrices(p, sd)
        Xd = sp.diags(sd.X)
        B = (Xd @ Ao @ Xd).toarray()
        ref = An.toarray() - sigma * B
        Sg, gd = s.local_matrix(j, 1)
        pos = np.searchsorted(sd.neu_dofs, gd)
        ref, B = ref[np.ix_(pos, pos)], B[np.ix_(pos, pos)]
        assert np.abs(Sg - ref).max() <= 1e-12 * np.abs(ref).max(), j
        Bg, _ = s.local_matrix(j, 2)
        assert np.abs(Bg - B).max() <= 1e-12 * np.abs(B).max(), j
    s.close()
