"""The variable-coefficient step on a grid whose planes in the library's chunks
exceed the 65535 chunks of a launch: one launch for all planes against the split
entry points, bit for bit."""
import pytest

from tests.gpu_util import lib, require_cuda

pytestmark = pytest.mark.gpu


# FP32 chunks hold 8 planes: the interior's 65535 chunks fit, all planes' 65536 do not
@pytest.mark.parametrize("dtype,nz", [("f32", 524280), ("f32", 524281), ("f32", 524282), ("f64", 524282)])
def test_all_planes_in_one_launch(dtype, nz):
    pkg, torch = lib(), require_cuda()
    u0 = torch.rand((nz, 1, 2), dtype=torch.float64, device="cuda",
                    generator=torch.Generator("cuda").manual_seed(1)).to(torch.float32 if dtype == "f32" else torch.float64)
    out = []
    for split in (False, True):
        with pkg.Heat(2, 1, nz, 1.0 / (12 * 0.95), dtype=dtype, flags=pkg.HS_VARKAPPA) as h:
            h.upload(u0)
            for _ in range(3):
                if split:
                    h.boundary(), h.interior(), h.swap()
                else:
                    h.step(1)
            out.append(h.read(torch.empty_like(u0)))
    assert torch.equal(out[0], out[1]) and not torch.equal(out[0], u0)
