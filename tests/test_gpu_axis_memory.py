"""The axis form's density quads (GPU): allocated for plans that take that form only,
replaced by the volume when there is no memory for them, with the same doses to
the bit, and allowed to come first inside a stream capture."""
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


def _plan():
    p = synth.small_plan(560, n=(23, 19, 17), vox=0.3, n_beams=3, field=3.0, couch=True, phantom="water")
    p.rho = np.random.default_rng(1).uniform(0.3, 1.7, p.rho.shape).astype(np.float32)
    return p


def test_other_forms_hold_no_quads(dc):
    import torch
    p = synth.small_plan(561, n=(160, 160, 160), vox=0.1, n_beams=1, field=1.0, phantom="water")

    def held(form):
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        plan = dc.dc_fspb_create_from(p, lateral_mode=form)
        used = free - torch.cuda.mem_get_info()[0]
        dc.dc_fspb_destroy(plan)
        return used
    held(dc.DC_LATERAL_AXIS)   # first use of the kernels
    # 16 bytes for each of 4.1 M voxels; the driver gives memory in pieces of 2 MiB
    assert held(dc.DC_LATERAL_AXIS) - held(dc.DC_LATERAL_ISO) >= 16 * 160**3 - 4 * 2**20


def test_same_doses_without_memory_for_the_quads(dc, monkeypatch):
    p = _plan()
    want = dc.dc_fspb_dose(dc.dc_fspb_create_from(p, lateral_mode=dc.DC_LATERAL_AXIS), p.fluence)
    plan = dc.dc_fspb_create_from(p)
    monkeypatch.setenv("DC_FSPB_FAIL_ALLOC_AT", "1")
    dc.dc_fspb_set_lateral_mode(plan, dc.DC_LATERAL_AXIS)
    monkeypatch.delenv("DC_FSPB_FAIL_ALLOC_AT")
    assert np.array_equal(dc.dc_fspb_dose(plan, p.fluence), want)
    dc.dc_fspb_set_density(plan, np.float32(0.8) * p.rho)
    other = dc.dc_fspb_create_from(p, lateral_mode=dc.DC_LATERAL_AXIS)
    dc.dc_fspb_set_density(other, np.float32(0.8) * p.rho)
    assert np.array_equal(dc.dc_fspb_dose(plan, p.fluence), dc.dc_fspb_dose(other, p.fluence))


def test_first_axis_form_inside_a_capture(dc):
    import torch
    p = _plan()
    want = dc.dc_fspb_dose(dc.dc_fspb_create_from(p, lateral_mode=dc.DC_LATERAL_AXIS), p.fluence).reshape(-1)
    stream = torch.cuda.Stream()
    plan = dc.dc_fspb_create_from(p, stream=stream.cuda_stream)
    dc.dc_fspb_pair_count(plan)
    fluence = torch.from_numpy(p.fluence).cuda()
    dose = torch.zeros(plan.n_voxels, device="cuda")
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        dc.dc_fspb_set_lateral_mode(plan, dc.DC_LATERAL_AXIS)
        dc.dc_fspb_dose(plan, fluence, dose)
    assert float(dose.abs().max()) == 0.0   # nothing has run yet
    graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(dose.cpu().numpy(), want)
