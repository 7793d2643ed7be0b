"""The coarse correction beside the local solves, on streams of the caller's.

It runs on a stream of the library's own between two events, so it has to see
what the caller queued before and must be done before the sum of both parts.  The
operator is the same sums in every case: with the launch shape pinned,
bit-identical to a plain call on the default stream.
"""
import numpy as np
import pytest

from workloads.laminate import make_block

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=[0, 1])
def solvers(request):
    import torch
    pkg = require_gpu()
    mp = pytest.MonkeyPatch()
    for k, v in (("CLUSTER", 2), ("ROWS", 0), ("STAGED", 0)):
        mp.setenv("GENEO_SCHWARZ_" + k, str(v))
    stream = torch.cuda.Stream()
    p = make_block(12, 8, 4, [0.0, 45.0, -45.0, 90.0], partition=(3, 2, 1, 1))
    out = []
    for st in (None, stream.cuda_stream):
        s = pkg.GeneoSolver(stream=st)
        s.assemble(p)
        s.setup(p, request.param)
        out.append(s)
    torch.cuda.synchronize()
    yield pkg, stream, out
    for s in out:
        s.close()
    mp.undo()


def _inputs(solvers, n):
    import torch
    _, _, (plain, _) = solvers
    g = torch.Generator(device="cuda").manual_seed(1)
    r = [torch.randn(plain.ndof, dtype=torch.float64, device="cuda", generator=g) for _ in range(n)]
    want = [plain.apply_preconditioner(v) for v in r]
    torch.cuda.synchronize()
    return r, want


def test_order_on_a_callers_stream(solvers):
    import torch
    pkg, stream, (_, s) = solvers
    r, want = _inputs(solvers, 4)
    buf, z = torch.zeros_like(r[0]), torch.zeros_like(r[0])
    got = []
    slow = torch.randn(4096, 4096, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        for v in r:                        # r arrives late, and is overwritten at once
            for _ in range(4):
                slow = torch.tanh(slow @ slow)
            buf.copy_(v)
            pkg.geneo_apply_preconditioner(s.ctx, buf, z)
            buf.fill_(float("nan"))
            got.append(z.clone())
            z.fill_(float("nan"))
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a, b)


def test_solves_agree(solvers):
    _, _, (plain, s) = solvers
    (u0, st0), (u1, st1) = plain.solve(tol=1e-8, max_it=500), s.solve(tol=1e-8, max_it=500)
    assert st0["iterations"] == st1["iterations"] and np.array_equal(u0, u1)
