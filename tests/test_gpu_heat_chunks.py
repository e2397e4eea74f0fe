"""Chunk lengths on small grids, which heat_step advances in one launch without
chunks: the tuner does not choose one there, and the split entry points, which
run the Interior kernel in chunks, give the same field for any length."""
import math

import numpy as np
import pytest

from tests.gpu_util import lib, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("arith", ["f64", "f32", "fixed64"])
def test_tuner_leaves_chunks_alone_where_there_are_none(arith, tmp_path):
    require_cuda()
    lib()
    from paper_2608_11882_gb300 import autotune
    assert math.isfinite(autotune._gpu_timer(arith, (33, 40, 70), 1, 1.0))
    assert autotune._gpu_timer(arith, (33, 40, 70), 1, 0.5) == math.inf
    assert math.isfinite(autotune._gpu_timer("f64", (180, 180, 180), 1, 0.5))
    t = autotune.Tuner(cache_path=tmp_path / "t.json", gpu_name="g")
    choice = t.best(arith, (33, 40, 70))
    assert choice["kc_factor"] == 1.0
    assert autotune.Tuner(cache_path=tmp_path / "t.json", gpu_name="g").best(arith, (33, 40, 70)) == choice


@pytest.mark.parametrize("arith", ["f64", "f32", "fixed64"])
@pytest.mark.parametrize("shape", [(1, 1, 1), (3, 9, 65), (10, 17, 129), (57, 33, 70), (24, 8, 64)])
def test_split_entry_points_in_chunks(arith, shape):
    pkg, torch = lib(), require_cuda()
    nz, ny, nx = shape
    dt = "f32" if arith == "f32" else "f64"
    flags = pkg.HS_FIXED64 if arith == "fixed64" else 0
    u0 = torch.from_numpy(np.random.default_rng(sum(shape)).uniform(-1, 1, size=shape)).cuda()
    u0 = u0.float() if dt == "f32" else u0
    with pkg.Heat(nx, ny, nz, 0.14, dtype=dt, flags=flags | pkg.HS_SCHED_FULL) as h:
        want = h.upload(u0).step(7).read(torch.empty_like(u0))
    for planes in (0, 1, 4, 5, 1000):
        with pkg.Heat(nx, ny, nz, 0.14, dtype=dt, flags=flags, tdepth=1) as h:
            h.kchunk = planes
            h.upload(u0)
            for _ in range(7):
                h.boundary(), h.interior(), h.swap()
            assert torch.equal(h.read(torch.empty_like(u0)), want), planes
