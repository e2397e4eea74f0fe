"""Which grids heat_step advances in one launch for all steps: those whose bricks
are few enough, thin grids (mostly empty bricks) among the others, with the same
result bit for bit either way."""
import numpy as np
import pytest

from tests.gpu_util import lib, require_cuda

pytestmark = pytest.mark.gpu


# (nz, ny, nx): on both sides of each line
@pytest.mark.parametrize("arith,shape,one", [
    ("f64", (160, 160, 160), True),
    ("f64", (900, 9, 500), True), ("f64", (310, 200, 66), False),          # 3600 and 3900 bricks
    ("f64", (400, 640, 16), False), ("f64", (176, 176, 176), False),
    ("fixed64", (400, 400, 20), True), ("fixed64", (380, 600, 17), False),
    ("f32", (128, 128, 128), True), ("f32", (144, 144, 144), False),       # 512 and 972 bricks, four deep
    ("f32", (140, 140, 250), True), ("f32", (120, 120, 370), False),       # 1260 and 1440, two deep
    ("f32", (260, 260, 60), True), ("f32", (370, 360, 60), False),         # thin, below and above 2^22 points
    ("f32", (600, 600, 20), True), ("f32", (340, 340, 65), False), ("f32", (10, 640, 640), True)])
def test_line_and_results(arith, shape, one):
    pkg, torch = lib(), require_cuda()
    from paper_2608_11882_gb300 import _native as native
    nz, ny, nx = shape
    dt = "f32" if arith == "f32" else "f64"
    flags = pkg.HS_FIXED64 if arith == "fixed64" else 0
    u0 = torch.from_numpy(np.random.default_rng(sum(shape)).uniform(-1, 1, size=shape)).cuda()
    u0 = u0.float() if dt == "f32" else u0
    out = []
    for extra in (0, pkg.HS_SCHED_FULL):
        with pkg.Heat(nx, ny, nz, 0.13, dtype=dt, flags=flags | extra) as h:
            h.upload(u0)
            before = native.launch_count()
            h.step(9)
            launches = native.launch_count() - before
            if not extra:
                assert (launches == 1) == one
            out.append(h.read(torch.empty_like(u0)))
    assert torch.equal(out[0], out[1])


def test_long_runs_are_cut_into_launches():
    """A launch holds the GPU for 1024 steps at most; the parts go on from one another."""
    pkg, torch = lib(), require_cuda()
    from paper_2608_11882_gb300 import _native as native
    u0 = torch.from_numpy(np.random.default_rng(2).uniform(-1, 1, size=(9, 11, 70))).cuda()
    out = []
    for extra in (0, pkg.HS_SCHED_FULL):
        with pkg.Heat(70, 11, 9, 0.02, flags=extra) as h:
            h.upload(u0)
            before = native.launch_count()
            h.step(2500)
            assert native.launch_count() - before == (2500 if extra else 3)
            out.append(h.read(torch.empty_like(u0)))
    assert torch.equal(out[0], out[1])
