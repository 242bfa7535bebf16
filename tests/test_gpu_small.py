"""Doses of plans with few work units (GPU), which a CTA per unit evaluates: equal
to the bit to the warp-per-unit paths that the batch of plans and the dose with
its matrix take, in every form (lateral factors, table layout, exponentials), for
windows from one beamlet to several rows and chunks of them, with non-finite
fluences; and the pair counts they leave behind."""
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


CASES = [dict(n=(9, 8, 7), vox=0.25, n_beams=1, field=0.5, roi=0.3),
         dict(n=(15, 16, 11), vox=0.25, n_beams=3, field=4.0, roi=2.0, couch=True),
         dict(n=(13, 10, 12), vox=0.3, n_beams=2, field=5.0, beamlet=0.125, roi=3.0),
         dict(n=(31, 29, 27), vox=0.25, n_beams=5, field=3.0, beamlet=0.25, roi=3.0)]


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("axis", [False, True])
@pytest.mark.parametrize("j", range(len(CASES)))
def test_same_bits_as_the_other_paths(dc, j, axis, bf16):
    p = synth.small_plan(500 + j, **CASES[j])
    plan = dc.dc_fspb_create_from(p, lateral_mode=dc.DC_LATERAL_AXIS if axis else dc.DC_LATERAL_ISO)
    if bf16:
        dc.dc_fspb_set_precision(plan, dc.DC_PRECISION_BF16)
    f = np.random.default_rng(j).uniform(0, 1, plan.n_beamlets).astype(np.float32)
    batch = dc.dc_fspb_batch_create([plan])
    for fluence in (f, np.where(np.arange(len(f)) % 5 == 2, np.float32(np.inf), f).astype(np.float32)):
        dose = dc.dc_fspb_dose(plan, fluence)
        for _ in range(2):
            assert np.array_equal(dose, dc.dc_fspb_dose(plan, fluence), equal_nan=True)
        assert np.array_equal(dose.reshape(-1), dc.dc_fspb_batch_dose(batch, [fluence])[0].reshape(-1), equal_nan=True)
        if not bf16:   # the matrix is always in FP32
            assert np.array_equal(dose.reshape(-1), dc.dc_fspb_dose_and_matrix(plan, fluence)[0].reshape(-1), equal_nan=True)
    assert np.isfinite(dc.dc_fspb_dose(plan, f)).all() and dc.dc_fspb_dose(plan, f).max() > 0
    assert dc.dc_fspb_pair_count(plan) == dc.dc_fspb_pair_count(dc.dc_fspb_create_from(p))
