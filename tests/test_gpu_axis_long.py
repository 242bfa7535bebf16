"""The axis form (GPU) on a grid of more than 2^23 voxels along an axis, where adding
2^23 no longer gives a tap's whole part: the doses from the density quads are those
from the volume, to the bit, at the far end as well."""
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


def test_far_end_of_a_long_axis(dc, monkeypatch):
    n, dx = (1 << 23) + 200, 1e-5
    g = synth.centred_grid(n, 2, 2, dx, 1.0, 1.0)
    rho = np.ones((2, 2, n), np.float32)
    rho[:, :, -400:] = np.random.default_rng(3).uniform(0.3, 1.7, (2, 2, 400))
    far = g.ox + (n - 1) * dx
    comm = synth.make_commissioning(roi_radius=0.6, smooth_sigma=1e-4, w_dt=0.125)
    p = synth.Plan("long", g, rho, [synth.Beam(0.0, 100.0, (far, 0.0, 0.0), 0.5, 0.5)], 0.5, 0.5, comm, np.ones(1, np.float32))
    with_quads = dc.dc_fspb_create_from(p, lateral_mode=dc.DC_LATERAL_AXIS)
    got = dc.dc_fspb_dose(with_quads, p.fluence)
    dc.dc_fspb_destroy(with_quads)
    plan = dc.dc_fspb_create_from(p)
    monkeypatch.setenv("DC_FSPB_FAIL_ALLOC_AT", "1")   # no memory for the quads
    dc.dc_fspb_set_lateral_mode(plan, dc.DC_LATERAL_AXIS)
    monkeypatch.delenv("DC_FSPB_FAIL_ALLOC_AT")
    want = dc.dc_fspb_dose(plan, p.fluence)
    assert want[:, :, -100:].min() > 0 and np.ptp(want[0, 0, -100:]) > 0
    assert np.array_equal(got, want)
