"""Where x += alpha p happens in solves of three kernels per iteration: in the
update pass for systems that stay in L2, in the direction pass for large ones
and for every system of a batch that holds a large one.  The values are the
same, so results agree bit for bit wherever the solve stops."""
import numpy as np
import pytest

from tests.gpu_util import lib, require_cuda
from workloads import cg_rhs, lap7_csr

pytestmark = pytest.mark.gpu


def operator(pkg, kind, shape):
    torch = require_cuda()
    nz, ny, nx = shape
    if kind == "stencil":
        return pkg.Operator.stencil(nx, ny, nz)
    return pkg.Operator.csr(*(torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in lap7_csr(nx, ny, nz)))


# odd and even counts of unknowns; a stencil below the one-launch sizes, a narrow
# one whose SpMV is staged (it tracks the direction's largest exponent)
@pytest.mark.parametrize("kind,shape", [("csr", (23, 17, 31)), ("csr", (40, 33, 26)), ("stencil", (24, 24, 24)),
                                        ("stencil", (100, 100, 8))])
@pytest.mark.parametrize("max_iter", [1, 2, 5, 36, 2000])
def test_alone_in_a_batch_and_beside_a_large_system(kind, shape, max_iter):
    pkg, torch = lib(), require_cuda()
    n = int(np.prod(shape))
    op, big = operator(pkg, kind, shape), operator(pkg, "stencil", (164, 160, 162))
    b, x0 = (torch.from_numpy(cg_rhs(n, seed=s)).cuda() for s in (4, 5))
    store = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
    store[1:] = x0
    with pkg.CG(op) as cg:
        x1, i1 = cg.run(b, x=x0.clone(), rtol=1e-6, max_iter=max_iter)
        x2, i2 = cg.run(b, x=store[1:], rtol=1e-6, max_iter=max_iter)   # x at an 8-byte address
    with pkg.CGBatch([op]) as cb:
        x3, i3 = cb.run([b], [x0.clone()], rtol=1e-6, max_iter=max_iter)
    bb = torch.from_numpy(cg_rhs(big.n, seed=6)).cuda()
    with pkg.CGBatch([big, op]) as cb:
        x4, i4 = cb.run([bb, b], [torch.zeros_like(bb), x0.clone()], rtol=1e-6, max_iter=max_iter)
    assert i1["iters"] == i2["iters"] == i3[0]["iters"] == i4[1]["iters"]
    assert i1["converged"] == (max_iter == 2000)
    assert torch.equal(x1, x2) and torch.equal(x1, x3[0]) and torch.equal(x1, x4[1])
    assert abs(i1["relres_recur"] - i1["relres_true"]) <= 1e-9 * max(1.0, i1["relres_true"])


@pytest.mark.parametrize("max_iter", [1, 2, 37, 2000])
def test_large_csr_keeps_two_directions(max_iter):
    """2^22 unknowns and up: CSR alone (two direction buffers) and in a batch (one)."""
    pkg, torch = lib(), require_cuda()
    op = operator(pkg, "csr", (162, 161, 163))
    b = torch.from_numpy(cg_rhs(op.n, seed=8)).cuda()
    with pkg.CG(op) as cg:
        x1, i1 = cg.run(b, rtol=1e-3, max_iter=max_iter)
    with pkg.CGBatch([op]) as cb:
        x2, i2 = cb.run([b], rtol=1e-3, max_iter=max_iter)
    assert i1["iters"] == i2[0]["iters"] and i1["converged"] == (max_iter == 2000)
    assert torch.equal(x1, x2[0])
    assert abs(i1["relres_recur"] - i1["relres_true"]) <= 1e-9 * max(1.0, i1["relres_true"])
