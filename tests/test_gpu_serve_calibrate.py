"""The k-bar model is fitted on the kernel that steps the server's requests."""
import numpy as np
import pytest

from tests.gpu_util import lib, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_prediction_matches_a_tick_alone(dtype):
    """Summed over 96^3 and 160^3, the prediction is within a factor of 1.5 of the
    device time of the server's own launch (the model's k is a mean over sizes
    whose costs per point differ less than that; heat_step differs 2 to 4 times)."""
    pkg, torch = lib(), require_cuda()
    from paper_2608_11882_gb300.serve import GpuBackend, Request, predict_seconds
    be = GpuBackend(workers=1)
    kbars = be.calibrate(edges=(96, 160))
    measured = predicted = 0.0
    for n in (96, 160):
        q = Request(n, "heat", (n, n, n), dtype, 0.1, 64,
                    payload=np.random.default_rng(n).uniform(-1, 1, (n, n, n)))
        h = be.heat_open(q)
        be.io_stream.synchronize()
        be.heat_advance([h], [4])
        with pkg.HeatBatch([h], [64], stream=be.stream) as b:
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(be.stream)
            b.run(use_graph=False)
            e1.record(be.stream)
            b.wait()
        measured += e0.elapsed_time(e1) * 1e-3
        predicted += predict_seconds(q, kbars)
        be.heat_close(h)
    be.close()
    assert 1 / 1.5 < predicted / measured < 1.5, (predicted, measured)
