"""Set-up workspaces do not outgrow what they were with FP64 tiles in both orders
(host-only, no GPU): a problem that filled the device then still fits.

The bounds are the estimates of the library that kept L and L^T of every FP64
factor and had no digits; the factors dominate them (16 bytes an entry of the
shifted Neumann matrices, 14 now that digits take the tiles' place).
"""
import pytest

import paper_1901_05188_gb300 as pkg
import workloads
from workloads.darcy import darcy_config

# (workload, precision): bytes
BOUND = {("tiny", 1): 2108248, ("small", 0): 35519832, ("small", 1): 32152408,
         ("c1", 0): 35432280, ("c1", 1): 32262488, ("c2", 0): 4139346776, ("c2", 1): 3500547416,
         ("c3", 0): 50488090200, ("c3", 1): 41593012824, ("d-small", 0): 19386968,
         ("d-small", 1): 16745560, ("d-large", 0): 1934177368, ("d-large", 1): 1496039512,
         ("d-spe10", 0): 15355705176, ("d-spe10", 1): 13185552216}


@pytest.mark.parametrize("name,prec", sorted(BOUND))
def test_set_up_workspace(name, prec):
    p = darcy_config(name) if name.startswith("d-") else workloads.config(name)
    keep = []
    _, need = pkg.geneo_estimate_workspace_bytes(
        pkg.GeneoSolver.mesh_of(p, keep), pkg.GeneoSolver.partition_of(p), pkg.GeneoSolver.modes_of(p),
        prec, pkg.GeneoSolver.unknowns_per_node(p))
    assert need <= BOUND[name, prec]
