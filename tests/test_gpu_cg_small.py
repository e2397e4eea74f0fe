"""Small matrix-free systems solved whole in one launch (2^14 to 2^22 unknowns):
against the oracle's operator and iteration count, and batch against single,
which run different kernels (several bricks per block, or one in registers)
with the same sums, bit for bit."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import lib, require_cuda
from workloads import cg_rhs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    oracle.build()
    return lib()


def dev(a):
    return require_cuda().from_numpy(np.ascontiguousarray(a)).cuda()


# bricks are 64 x 8 x 4 or 32 x 16 x 4 points: exact fits, one past an edge per
# axis, odd rows (padded vectors), narrow rows, one block per brick and several
SHAPES = [(32, 32, 64), (33, 17, 65), (29, 31, 33), (64, 64, 16), (40, 50, 17), (5, 63, 127), (101, 90, 131),
          (128, 128, 128)]


@pytest.mark.parametrize("shape", SHAPES)
def test_against_oracle_and_batch(pkg, shape):
    nz, ny, nx = shape
    n = nx * ny * nz
    rtol = 1e-8
    b = cg_rhs(n, seed=sum(shape))
    _, ref = oracle.cg_solve(b, rtol, 5000, shape=shape, threads=oracle.max_threads())
    op = pkg.Operator.stencil(nx, ny, nz)
    with pkg.CG(op) as cg:
        x, info = cg.run(dev(b), rtol=rtol, max_iter=5000)
        again, _ = cg.run(dev(b), rtol=rtol, max_iter=5000)
    xh = x.cpu().numpy()
    assert info["converged"] and abs(info["iters"] - ref["iters"]) <= 2
    r = b - oracle.lap7_apply(xh.reshape(shape), threads=oracle.max_threads()).reshape(-1)
    res = np.linalg.norm(r) / np.linalg.norm(b)
    assert res <= 1.5 * rtol and abs(info["relres_true"] - res) <= 1e-3 * rtol
    assert np.array_equal(again.cpu().numpy(), xh)
    other = pkg.Operator.stencil(30, 28, 26)
    with pkg.CGBatch([other, op]) as cb:
        xs, infos = cb.run([dev(cg_rhs(30 * 28 * 26, seed=1)), dev(b)], rtol=rtol, max_iter=5000)
    assert np.array_equal(xs[1].cpu().numpy(), xh) and infos[1]["iters"] == info["iters"]
    assert infos[1]["relres_true"] == info["relres_true"] and infos[0]["converged"]


@pytest.mark.parametrize("nx", [32, 33])
def test_start_vector_limits_and_zero_rhs(pkg, nx):
    """A start vector at an 8-byte address, max_iter, rtol met at once, a zero
    right-hand side, and vectors scaled outside the exact-sum range."""
    torch = require_cuda()
    ny, nz = 31, 30
    n = nx * ny * nz
    b = dev(cg_rhs(n, seed=5))
    store = torch.zeros(n + 1, dtype=torch.float64, device="cuda")
    with pkg.CG(pkg.Operator.stencil(nx, ny, nz)) as cg:
        x1, i1 = cg.run(b, rtol=1e-10)
        x2, i2 = cg.run(b, x=store[1:], rtol=1e-10)
        assert i1["iters"] == i2["iters"] and torch.equal(x1, x2)
        x3, i3 = cg.run(b, x=x1.clone(), rtol=1e-9)
        assert i3["iters"] == 0 and i3["converged"] and torch.equal(x3, x1)
        _, i4 = cg.run(b, rtol=1e-12, max_iter=7)
        assert i4["iters"] == 7 and not i4["converged"]
        assert abs(i4["relres_recur"] - i4["relres_true"]) <= 1e-10 * i4["relres_true"]
        x5, i5 = cg.run(torch.zeros_like(b), x=torch.ones_like(b), rtol=1e-8)
        assert i5["converged"] and i5["iters"] == 0 and not x5.any()
        x6, i6 = cg.run(b * 2.0 ** -500, rtol=1e-8)   # p's exponent leaves the range, its square does not underflow
        assert i6["converged"] and i6["relres_true"] <= 1.5e-8


def test_more_systems_than_one_group(pkg):
    """70 systems: two groups of one launch, with a zero right-hand side and
    systems that stop at very different iterations."""
    rng = np.random.default_rng(9)
    shapes = [tuple(int(v) for v in rng.integers(26, 34, 3)) for _ in range(70)]
    bs = [cg_rhs(int(np.prod(s)), seed=i) for i, s in enumerate(shapes)]
    bs[11][:] = 0.0
    ops = [pkg.Operator.stencil(*s[::-1]) for s in shapes]
    with pkg.CGBatch(ops) as cb:
        xs, infos = cb.run([dev(b) for b in bs], rtol=1e-9, max_iter=500)
    assert all(i["converged"] for i in infos)
    for k in (0, 11, 40, 69):
        with pkg.CG(ops[k]) as cg:
            x1, i1 = cg.run(dev(bs[k]), rtol=1e-9, max_iter=500)
        assert np.array_equal(xs[k].cpu().numpy(), x1.cpu().numpy()) and infos[k]["iters"] == i1["iters"]


# one block per brick, several bricks per block, and fewer unknowns than either takes
@pytest.mark.parametrize("shape", [(32, 32, 64), (33, 17, 65), (128, 128, 128), (12, 20, 18)])
def test_overflowing_pq_ends_at_max_iter(pkg, shape):
    """||r||^2 finite and p.q beyond the largest double: alpha is 0, x stays, and
    the solve ends at max_iter, alone and in a batch beside a system that goes on
    or converges.  r stays too, so p_i = (i + 1) r: the iterations are few enough
    that no single product p[k] q[k] overflows, which would make p.q NaN."""
    torch = require_cuda()
    nz, ny, nx = shape
    n = nx * ny * nz
    b = cg_rhs(n, seed=3)
    b /= np.linalg.norm(b)
    p2 = b.reshape(shape)
    its = 6
    assert float((p2 * oracle.lap7_apply(p2)).sum()) > 4.0                     # p.q > 2.4e308
    assert 12.0 * its ** 2 * float(np.abs(b).max()) ** 2 * 6e307 < 1.7e308     # |p[k] q[k]| of the last iteration
    b *= np.sqrt(6e307)
    x0 = torch.zeros(n, dtype=torch.float64, device="cuda")
    op, other = pkg.Operator.stencil(nx, ny, nz), pkg.Operator.stencil(30, 28, 26)
    bo = dev(cg_rhs(30 * 28 * 26, seed=1))
    with pkg.CG(op) as cg, pkg.CG(other) as co:
        x, info = cg.run(dev(b), x=x0.clone(), rtol=0.5, max_iter=its)
        xo, io = co.run(bo, rtol=0.5, max_iter=its)
    assert not info["converged"] and info["iters"] == its and torch.equal(x, x0)
    assert abs(info["relres_recur"] - 1.0) < 1e-12 and abs(info["relres_true"] - 1.0) < 1e-12
    assert io["converged"] and io["iters"] < its
    for ops, bs, k in (([op, other], [dev(b), bo], 0), ([other, op], [bo, dev(b)], 1)):
        with pkg.CGBatch(ops) as cb:
            xs, infos = cb.run(bs, rtol=0.5, max_iter=its)
            assert not infos[k]["converged"] and infos[k]["iters"] == its and torch.equal(xs[k], x0)
            assert infos[1 - k]["converged"] and torch.equal(xs[1 - k], xo)
            xs, infos = cb.run(bs, rtol=1e-8, max_iter=its)
            assert [i["iters"] for i in infos] == [its, its] and torch.equal(xs[k], x0)


@pytest.mark.parametrize("shape", [(32, 32, 64), (128, 128, 128), (12, 20, 18)])
@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_right_hand_side_that_is_not_finite(pkg, shape, bad):
    """A breakdown, alone and in a batch, and the context solves on."""
    nz, ny, nx = shape
    b = cg_rhs(nx * ny * nz, seed=3)
    poisoned = b.copy()
    poisoned[nx * ny + 5] = bad
    op, other = pkg.Operator.stencil(nx, ny, nz), pkg.Operator.stencil(30, 28, 26)
    bo = dev(cg_rhs(30 * 28 * 26, seed=1))
    with pkg.CG(op) as cg, pkg.CGBatch([other, op]) as cb:
        with pytest.raises(Exception, match="breakdown"):
            cg.run(dev(poisoned), max_iter=40)
        with pytest.raises(Exception, match="breakdown in system 1"):
            cb.run([bo, dev(poisoned)], max_iter=40)
        x, info = cg.run(dev(b), rtol=1e-6, max_iter=2000)
        xs, infos = cb.run([bo, dev(b)], rtol=1e-6, max_iter=2000)
    assert info["converged"] and infos[0]["converged"] and np.array_equal(xs[1].cpu().numpy(), x.cpu().numpy())
