"""The multi-step kernel (all steps of a small grid in one cooperative launch)
against the one-kernel full step (HS_SCHED_FULL), whose per-point arithmetic is
the same: equal bit for bit."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import F64_REL, lib, rel_max_err, require_cuda

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    oracle.build()
    return lib()


def flag(pkg, arith):
    return pkg.HS_FIXED64 if arith == "fixed64" else 0


# bricks are 64 x 8 x 4 points (FP32 64 x 16 x 4): one point, one short of an
# edge, an edge, one past it, per axis; a grid of several bricks per block
@pytest.mark.parametrize("shape", [(1, 1, 1), (4, 8, 64), (3, 7, 63), (5, 9, 65), (5, 17, 129), (4, 16, 128),
                                   (61, 37, 45), (101, 90, 131), (2, 300, 200), (160, 160, 163)])
@pytest.mark.parametrize("arith", ["f64", "f32", "fixed64"])
def test_equals_full_step_kernel(pkg, arith, shape):
    nz, ny, nx = shape
    dt = "f32" if arith == "f32" else "f64"
    u0 = np.random.default_rng(sum(shape)).uniform(-1, 1, size=shape).astype(np.float32 if dt == "f32" else np.float64)
    out = []
    for extra, parts in ((0, (1, 5, 2)), (pkg.HS_SCHED_FULL, (8,))):
        with pkg.Heat(nx, ny, nz, 0.13, dtype=dt, flags=flag(pkg, arith) | extra) as h:
            h.upload(u0)
            for n in parts:
                h.step(n)
            assert h.steps_done == 8
            out.append(h.read())
    assert np.array_equal(out[0], out[1])
    if arith == "f64":
        assert rel_max_err(out[0], oracle.heat_run(u0, 0.13, 8, threads=oracle.max_threads())) <= F64_REL


@pytest.mark.parametrize("arith", ["f64", "fixed64"])
def test_scale_follows_a_shrinking_field(pkg, arith):
    """The step maximum changes its exponent many times (a 20 x 9 x 6 grid loses
    about 6% per step), also between the kernels that share its record."""
    u0 = np.random.default_rng(3).uniform(0.5, 1, size=(6, 9, 20))
    out = []
    for extra in (0, pkg.HS_SCHED_FULL):
        with pkg.Heat(20, 9, 6, 0.16, flags=flag(pkg, arith) | extra) as h:
            h.upload(u0).step(150)
            for _ in range(3):   # the split entry points go on from the multi-step kernel's record
                h.boundary(), h.interior(), h.swap()
            h.step(150)
            out.append(h.read())
    assert np.array_equal(out[0], out[1])
    assert 0 < np.max(np.abs(out[0])) < 1e-5


def test_captured_steps_replay(pkg):
    """heat_step under stream capture: six steps (a multiple of both buffer and
    maximum-record periods) replayed three times after six direct ones."""
    torch = require_cuda()
    u0 = np.random.default_rng(5).uniform(-1, 1, size=(33, 40, 70))
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        h = pkg.Heat(70, 40, 33, 0.15)
        h.upload(u0).step(6)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            h.step(6)
        for _ in range(3):
            g.replay()
        got = h.read()
        h.close()
    with pkg.Heat(70, 40, 33, 0.15, flags=pkg.HS_SCHED_FULL) as f:
        assert np.array_equal(got, f.upload(u0).step(24).read())
