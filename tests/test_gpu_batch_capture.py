"""Several fluence vectors inside a stream capture (GPU): once a call of as many
vectors has been made, in either precision, the FP32 form allocates nothing more,
so it can be captured and replayed."""
import numpy as np
import pytest

from paper_1103_1164_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dc():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1103_1164_gb300 import build, dc_fspb
    build.build()
    dc_fspb.load()
    return dc_fspb


@pytest.mark.parametrize("first", ["DC_PRECISION_FP32", "DC_PRECISION_BF16"])
@pytest.mark.parametrize("k", [7, 20, 64])
def test_fp32_batch_in_a_capture(dc, k, first):
    import torch
    p = synth.small_plan(570, n=(23, 19, 17), vox=0.3, n_beams=3, field=3.0, couch=True)
    F = np.random.default_rng(k).uniform(0, 1, (k, p.n_beamlets)).astype(np.float32)
    want = dc.dc_fspb_dose_batch(dc.dc_fspb_create_from(p), F).reshape(k, -1)
    stream = torch.cuda.Stream()
    plan = dc.dc_fspb_create_from(p, stream=stream.cuda_stream)
    fluence = torch.from_numpy(F).cuda()
    dose = torch.zeros((k, plan.n_voxels), device="cuda")
    torch.cuda.synchronize()
    dc.dc_fspb_set_precision(plan, getattr(dc, first))
    dc.dc_fspb_dose_batch(plan, fluence, dose)
    dc.dc_fspb_set_precision(plan, dc.DC_PRECISION_FP32)
    dc.dc_fspb_device_status(plan)
    dose.zero_()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        dc.dc_fspb_dose_batch(plan, fluence, dose)
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(dose.cpu().numpy(), want)
