"""The direction pass of large solves, which keeps two direction buffers and
adds two iterations' steps to x at once, against the batched solve, which adds
one at a time in place: equal bit for bit wherever the solve stops."""
import numpy as np
import pytest

from tests.gpu_util import lib, require_cuda
from workloads import cg_rhs

pytestmark = pytest.mark.gpu


# 2^22 unknowns and up; an odd count of unknowns (177) takes the scalar tail
@pytest.mark.parametrize("shape", [(164, 160, 162), (161, 159, 177)])
@pytest.mark.parametrize("max_iter", [1, 2, 3, 36, 37, 5000])
def test_stops_at_any_iteration(shape, max_iter):
    pkg, torch = lib(), require_cuda()
    nz, ny, nx = shape
    n = nx * ny * nz
    assert n >= 1 << 22
    op = pkg.Operator.stencil(nx, ny, nz)
    b = torch.from_numpy(cg_rhs(n, seed=8)).cuda()
    x0 = torch.from_numpy(cg_rhs(n, seed=9)).cuda()
    store = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
    with pkg.CG(op) as cg:
        x1, i1 = cg.run(b, x=x0.clone(), rtol=1e-3, max_iter=max_iter)
        store[1:] = x0
        x2, i2 = cg.run(b, x=store[1:], rtol=1e-3, max_iter=max_iter)   # x at an 8-byte address
    with pkg.CGBatch([op]) as cb:
        x3, i3 = cb.run([b], [x0.clone()], rtol=1e-3, max_iter=max_iter)
    assert i1["iters"] == i2["iters"] == i3[0]["iters"]
    assert i1["converged"] == (max_iter == 5000)
    assert torch.equal(x1, x2) and torch.equal(x1, x3[0])
    assert abs(i1["relres_recur"] - i1["relres_true"]) <= 1e-9 * max(1.0, i1["relres_true"])
