"""Batched local solves with a cluster of CTAs per (instance, subdomain) item.

The cluster splits the tiles of a row over its CTAs and leaves the operator as
it is, so every launch shape solves the same systems with sums in another
order: FP64 solutions within 1e-9 of the one-CTA shape's and iterations within
one, the bounds that hold between batched and single solves; with FP32 factors
both are within 1e-6 of the solution at tol 1e-10, iterations within two.  The
instances go from one tile row per subdomain to more rows than a cluster has
tiles for, with half-bandwidths below and above the cluster size.
"""
import pytest

import workloads
from workloads.darcy import darcy_config
from workloads.laminate import make_block

from gpu_common import rel, require_gpu

pytestmark = pytest.mark.gpu


def _solve(pkg, prec, monkeypatch, shape):
    for k, v in zip(("CLUSTER", "ROWS", "STAGED"), shape):
        monkeypatch.setenv("GENEO_SCHWARZ_" + k, str(v))
    thr = dict(fixed_modes=0, threshold=0.0, max_modes=20, shift=-0.01)
    solvers = []
    for p in (workloads.config("tiny"), workloads.config("small"),
              make_block(10, 6, 4, [0.0, 90.0, 90.0, 0.0], partition=(3, 2, 1, 1), modes=thr),
              make_block(14, 4, 3, [45.0, -45.0, -45.0], partition=(4, 1, 1, 1), modes=thr),
              darcy_config("d-tiny")):
        s = pkg.GeneoSolver()
        s.assemble(p)
        s.setup(p, prec)
        solvers.append(s)
    batch = pkg.GeneoBatch(solvers)
    us, stats = batch.solve(tol=1e-10 if prec else 1e-8, max_it=3000)
    batch.close()
    for s in solvers:
        s.close()
    return us, stats


@pytest.mark.parametrize("staged", [0, 1])
@pytest.mark.parametrize("rows", [0, 1])
@pytest.mark.parametrize("prec", [0, 1])
def test_batch_clusters_agree(monkeypatch, prec, rows, staged):
    pkg = require_gpu()
    one, st1 = _solve(pkg, prec, monkeypatch, (1, rows, staged))
    for cluster in (2, 4):
        us, stats = _solve(pkg, prec, monkeypatch, (cluster, rows, staged))
        for u, v, a, b in zip(us, one, stats, st1):
            assert (a["schwarz_cluster"], a["schwarz_rows"], a["schwarz_staged"]) == (cluster, rows, staged)
            assert abs(a["iterations"] - b["iterations"]) <= (2 if prec else 1)
            assert rel(u, v) <= (2e-6 if prec else 1e-9)
