"""FP32 temporal blocking around the edges of its tiles -- 120 columns (one warp
per row, x neighbours by lane shuffle) or 128 (rows of 34 threads), 28, 26 or
24 rows at depths 2, 3 and 4 -- and the library's choice of passes on grids
past the multi-step kernel: the one-step kernels' field bit for bit."""
import numpy as np
import pytest

from tests.gpu_util import lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    return lib()


def run(pkg, u0, steps, tdepth):
    nz, ny, nx = u0.shape
    with pkg.Heat(nx, ny, nz, 0.15, dtype="f32", tdepth=tdepth, flags=pkg.HS_SCHED_FULL if tdepth == 1 else 0) as h:
        h.upload(u0)
        h.step(steps)
        assert h.steps_done == steps
        return h.read()


def field(shape):
    return np.random.default_rng(sum(shape)).uniform(-1, 1, size=shape).astype(np.float32)


@pytest.mark.parametrize("tdepth", [2, 3, 4])
@pytest.mark.parametrize("shape", [(9, 28, 120), (20, 29, 121), (33, 27, 119), (5, 57, 241), (40, 24, 128),
                                   (17, 53, 256), (6, 25, 129), (70, 31, 361), (1, 1, 1)])
def test_tile_edges(pkg, shape, tdepth):
    u0 = field(shape)
    assert np.array_equal(run(pkg, u0, 13, 1), run(pkg, u0, 13, tdepth))


# 2^23 points and more: 120-column tiles (passes of four steps), 128-column
# tiles (passes of two); flat and tall grids
@pytest.mark.parametrize("shape", [(204, 203, 205), (129, 261, 256), (3, 1300, 2200), (2100, 62, 67)])
@pytest.mark.parametrize("steps", [1, 2, 3, 7, 12])
def test_library_choice(pkg, shape, steps):
    u0 = field(shape)
    with pkg.Heat(shape[2], shape[1], shape[0], 0.15, dtype="f32") as h:
        assert h.tdepth == 2
    assert np.array_equal(run(pkg, u0, steps, 1), run(pkg, u0, steps, 0))


@pytest.mark.parametrize("tdepth", [2, 4])
def test_very_tall_grid(pkg, tdepth):
    """More planes than 65535 chunks of the usual length hold."""
    u0 = field((8_600_000, 1, 1))
    assert np.array_equal(run(pkg, u0, 5, 1), run(pkg, u0, 5, tdepth))
