"""The exact-sum FP64 streaming kernel takes four planes per turn of its loop,
each turn with the ring's slots and the two register sets in fixed places:
chunks of every remainder modulo four and shorter than one turn, grids whose
tiles are cut in x and y, and the default chunk of the plane-count rule."""
import numpy as np
import pytest

import oracle
from tests.gpu_util import F64_REL, lib
from workloads import heat_u0_single_mode

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    oracle.build()
    return lib()


# 2^22 points and more (smaller grids take the multi-step kernel)
@pytest.mark.parametrize("shape", [(163, 161, 162), (39, 250, 437), (260, 131, 129)])
@pytest.mark.parametrize("scale", [1.0, 1e-310])   # fixed point; the FP64-pipe form
def test_every_chunk_remainder(pkg, shape, scale):
    nz, ny, nx = shape
    u0 = heat_u0_single_mode(nx, ny, nz, seed=23) * scale
    ref = oracle.heat_run(u0, 1.0 / 7, 3, threads=oracle.max_threads())
    # the FP64 form at 1e-310: subnormal values, each operation off by up to half a unit
    bound = F64_REL * float(np.max(np.abs(ref))) + (8 * 3 * 2.0 ** -1074 if scale != 1.0 else 0.0)
    first = None
    for kc in (None, 1, 2, 3, 4, 5, 6, 7, 8, 9, nz):
        with pkg.Heat(nx, ny, nz, 1.0 / 7) as h:
            if kc is not None:
                h.kchunk = kc
            h.upload(u0)
            h.step(3)
            got = h.read()
        assert float(np.max(np.abs(got - ref))) <= bound, kc
        first = got if first is None else first
        assert np.array_equal(got, first), kc
