"""What admission counts for a request covers what the library allocates for it."""
import ctypes

import pytest

from paper_2608_11882_gb300 import _native as nat
from paper_2608_11882_gb300.serve import Request, device_bytes


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("shape", [(1, 1, 1), (8, 8, 8), (61, 37, 45), (64, 64, 64), (5, 3, 127)])
def test_heat_covers_the_handle(dtype, shape):
    nz, ny, nx = shape
    desc = nat.hs_heat_desc(nx=nx, ny=ny, nz=nz, r=0.1, flags=0, dtype=nat.HS_F32 if dtype == "f32" else nat.HS_F64,
                            tdepth=1, stream=None)
    one = ctypes.c_size_t()
    assert nat.lib.heat_buffer_bytes(ctypes.byref(desc), ctypes.byref(one)) == 0
    # two buffers, each from a 256-byte boundary, after the handle's 1 KiB of words
    want = 1024 + 2 * ((one.value + 255) // 256 * 256)
    assert device_bytes(Request(0, "heat", shape, dtype)) == want


@pytest.mark.parametrize("shape,vectors,row", [
    ((20, 20, 20), 5, 20), ((64, 64, 65), 5, 66),          # an odd row of the one-launch solve is padded by one
    ((9000, 3, 1), 5, 1), ((128, 128, 15), 5, 15),         # narrow rows take the other solver, unpadded
    ((160, 160, 163), 5, 164), ((256, 256, 256), 6, 256), ((164, 160, 163), 6, 163)])
def test_cg_covers_the_vectors(shape, vectors, row):
    """b and x dense; r, q, p and from 2^22 unknowns a second p, padded or not;
    the partials of 4096 bricks and the control words."""
    nz, ny, nx = shape
    want = 8 * (2 * nx + (vectors - 2) * row) * ny * nz + 2 * 4096 * 8 + 2048
    got = device_bytes(Request(0, "cg", shape))
    assert want <= got <= want + 4096
