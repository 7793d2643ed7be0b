"""Batches whose local vectors nearly fill shared memory.

A batch holds every local vector whole in shared memory, and the exchange
buffers grow with the cluster: 227 KB less the queue's item leave an FP64 vector
883 - 2 C tile rows in a cluster of C.  880 rows fit one CTA, and with two fill the
227 KB to the byte, which leaves no room for the item; 876 do so with four.  A pinned cluster that does not fit is halved until one does, and
8, which a batch has not, means its largest: a pin neither refuses a batch nor
leaves the shape, and with it the order of the sums, to a timing.
"""
import numpy as np
import pytest

from workloads.darcy import make_darcy
from workloads.laminate import make_block

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

# (elements, unknowns of the largest subdomain, largest cluster that holds it)
SIZES = [((21, 78, 31), 28160, 1), ((25, 70, 29), 28080, 2), ((25, 68, 30), 28210, 0),
         ((19, 72, 37), 28120, 2),
         ((21, 96, 25), 28028, 2)]


def _solve(pkg, size, unknowns, monkeypatch, pins):
    p = make_darcy(*size, seed=4, partition=(1, 2, 1, 1))
    keep = []
    plan = pkg.geneo_plan_subdomains(pkg.GeneoSolver.mesh_of(p, keep), pkg.GeneoSolver.partition_of(p),
                                     unknowns_per_node=1)
    assert plan[:, 12].max() == unknowns
    s = pkg.GeneoSolver()
    s.assemble(p)
    s.setup(p, pkg.GENEO_FP64, pkg.GENEO_AS, pkg.GENEO_COARSE_NONE)
    for k, v in pins.items():
        monkeypatch.setenv("GENEO_SCHWARZ_" + k, v)
    try:
        batch = pkg.GeneoBatch([s])
        us, st = batch.solve(tol=1e-6, max_it=5000)
        batch.close()
    finally:
        s.close()
    assert np.all(np.isfinite(us[0])) and st[0]["rel_res_true"] <= 1e-5
    return st[0]["schwarz_cluster"]


@pytest.mark.parametrize("size,unknowns,most", SIZES)
def test_unpinned(monkeypatch, size, unknowns, most):
    pkg = require_gpu()
    if most:
        assert _solve(pkg, size, unknowns, monkeypatch, {}) <= most
    else:                                  # 882 rows: no launch holds them
        with pytest.raises(pkg.GeneoError) as e:
            _solve(pkg, size, unknowns, monkeypatch, {})
        assert e.value.status == 1         # GENEO_ERR_INVALID_ARG


@pytest.mark.parametrize("size,unknowns,most", [c for c in SIZES if c[2]])
@pytest.mark.parametrize("pin", [1, 2, 4, 8])
def test_a_pin_that_does_not_fit(monkeypatch, size, unknowns, most, pin):
    got = _solve(require_gpu(), size, unknowns, monkeypatch, {"CLUSTER": str(pin)})
    assert got == min(most, pin)


@pytest.mark.parametrize("pin,want", [(1, 1), (2, 2), (4, 4), (8, 4)])
def test_a_pin_that_fits(monkeypatch, pin, want):
    pkg = require_gpu()
    s = pkg.GeneoSolver()
    p = make_block(8, 6, 4, [0.0, 90.0, 90.0, 0.0], partition=(2, 1, 1, 1))
    s.assemble(p)
    s.setup(p, pkg.GENEO_FP64)
    for k, v in (("CLUSTER", pin), ("ROWS", 0), ("STAGED", 0)):
        monkeypatch.setenv("GENEO_SCHWARZ_" + k, str(v))
    batch = pkg.GeneoBatch([s])
    _, st = batch.solve()
    assert [st[0]["schwarz_" + k] for k in ("cluster", "rows", "staged")] == [want, 0, 0]
    batch.close()
    s.close()
