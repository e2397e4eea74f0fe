"""Where x += alpha p happens in solves of three kernels per iteration: in the
update pass for systems that stay in L2, in the direction pass for large ones
and for every system of a batch that holds a large one.  The values are the
same, so results agree bit for bit wherever the solve stops."""
import os
import subprocess
import sys

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


# a process of its own: its memory pool holds nothing from other solves
ONE_BUFFER = """
import torch, paper_2608_11882_gb300 as pkg
n = 400
op = pkg.Operator.stencil(n, n, n)
b = torch.randn(n ** 3, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
out = []
for its in (1, 6, 7):
    x = torch.zeros_like(b)
    with pkg.CG(op) as cg:
        out.append((x, cg.run(b, x, rtol=1e-3, max_iter=its)[1]))
vec = 8 * n ** 3
second = [torch.zeros_like(b) for _ in out]
torch.cuda.synchronize()
torch.cuda.empty_cache()
fill = torch.empty(torch.cuda.mem_get_info()[0] - 7 * vec // 2, dtype=torch.uint8, device="cuda")
assert 3 * vec < torch.cuda.mem_get_info()[0] < 4 * vec
for its, x, (x0, i0) in zip((1, 6, 7), second, out):
    with pkg.CG(op) as cg:
        _, info = cg.run(b, x, rtol=1e-3, max_iter=its)
    assert torch.equal(x, x0) and info == i0 and info["iters"] == its, (info, i0)
print("same")
"""


def test_one_direction_buffer_where_memory_is_short():
    """Room for r, q and one direction: the solve keeps one buffer and gives the
    same result bit for bit."""
    torch = require_cuda()
    lib()
    if torch.cuda.mem_get_info()[0] < 24 << 30:
        pytest.skip("needs 24 GB of device memory")
    torch.cuda.empty_cache()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", ONE_BUFFER], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.split() == ["same"], r.stderr[-2000:]
