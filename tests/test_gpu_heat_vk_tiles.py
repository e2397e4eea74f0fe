"""The FP64 variable-coefficient kernel (tiles of 64 x 8 columns, a ring of
staged planes, fluxes in integers) at the sizes where its tiling can go wrong,
and its three ways through a step."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import lib, rel_max_err

pytestmark = pytest.mark.gpu

R = 1.0 / (12 * 0.95)


@pytest.fixture(scope="module")
def pkg():
    oracle.build()
    return lib()


# per step: fluxes and sum within 30 2^-57 max|u| beta, the oracle's formula within
# about 24 roundings of terms below 12 1.9 max|u| beta (beta = 0.044), plus the
# rounding of each result and of dt f: under 6e-16 of max|u|
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 8, 64), (3, 7, 63), (4, 9, 65), (5, 17, 129), (33, 16, 128),
                                   (70, 70, 70), (1, 40, 33)])
def test_tile_edges_against_oracle(pkg, shape):
    nz, ny, nx = shape
    u0 = np.random.default_rng(sum(shape)).uniform(-1, 1, size=shape)
    ref = oracle.heat_vk_run(u0, R, 12, threads=oracle.max_threads())
    with pkg.Heat(nx, ny, nz, R, flags=pkg.HS_VARKAPPA) as h:
        got = h.upload(u0).step(12).read()
    assert rel_max_err(got, ref) <= 12 * 6e-16 * np.max(np.abs(u0)) / np.max(np.abs(ref))


@pytest.mark.parametrize("shape", [(21, 19, 70), (20, 20, 20)])
def test_parts_chunks_and_timing_change_nothing(pkg, shape):
    """Boundary + Interior + swap, any planes per block, and the timed schedule
    give the one-launch step bit for bit; so does a field whose scale leaves the
    integer form's range and comes back (the FP64 formula in between)."""
    nz, ny, nx = shape
    u0 = np.random.default_rng(4).uniform(-1, 1, size=shape)
    out = []
    for how in ("step", "parts", "chunk1", "chunk7", "timed"):
        with pkg.Heat(nx, ny, nz, R, flags=pkg.HS_VARKAPPA) as h:
            h.upload(u0)
            if how.startswith("chunk"):
                h.kchunk = int(how[5:])
            if how == "timed":
                h.time_interior(True)
            for _ in range(5):
                if how == "parts":
                    h.boundary(), h.interior(), h.swap()
                else:
                    h.step(1)
            out.append(h.read())
    for o in out[1:]:
        assert np.array_equal(o, out[0])
    tiny = u0 * 1e-300
    ref = oracle.heat_vk_run(tiny, R, 8)
    with pkg.Heat(nx, ny, nz, R, flags=pkg.HS_VARKAPPA) as h:
        assert rel_max_err(h.upload(tiny).step(8).read(), ref) <= 1e-13
