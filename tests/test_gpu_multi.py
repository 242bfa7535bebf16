"""Several fluence vectors in one pass (GPU): every pass width, at its first and
last number of vectors, against the single-vector dose, with merged and general
tables and per-entry lateral factors, windows shorter and longer than the
staged chunk, and fluences that are not finite (which reach the beamlet's own
voxels only)."""
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


CASES = [dict(n=(21, 19, 17), vox=0.25, n_beams=3, field=3.0, roi=1.0),
         dict(n=(17, 23, 12), vox=0.3, n_beams=2, field=2.0, roi=3.0),
         dict(n=(15, 14, 13), vox=0.35, n_beams=2, field=5.0, beamlet=0.25, roi=4.0, couch=True)]


def _plan(dc, j, axis):
    return dc.dc_fspb_create_from(synth.small_plan(700 + j, **CASES[j]),
                                  lateral_mode=dc.DC_LATERAL_AXIS if axis else dc.DC_LATERAL_ISO)


@pytest.mark.parametrize("axis", [False, True])
@pytest.mark.parametrize("j", range(len(CASES)))
def test_equals_single_vectors(dc, j, axis):
    plan = _plan(dc, j, axis)
    F = np.random.default_rng(j).uniform(0, 1, (64, plan.n_beamlets)).astype(np.float32)
    one = np.stack([dc.dc_fspb_dose(plan, np.ascontiguousarray(f)) for f in F])
    for k in (2, 16, 17, 32, 33, 64):
        got = dc.dc_fspb_dose_batch(plan, np.ascontiguousarray(F[:k]))
        # the same sums over the same pairs in the same order
        assert np.abs(got - one[:k]).max() <= 1e-6 * one.max(), k


@pytest.mark.parametrize("k", [3, 20, 64])
def test_non_finite_fluence_stays_with_its_beamlet(dc, k):
    plan = _plan(dc, 0, False)
    F = np.random.default_rng(k).uniform(0, 1, (k, plan.n_beamlets)).astype(np.float32)
    F[0, 7], F[1, 20], F[k - 1, plan.n_beamlets - 1] = np.inf, np.nan, -np.inf
    got = dc.dc_fspb_dose_batch(plan, F)
    for q in (0, 1, 2, k - 1):
        one = dc.dc_fspb_dose(plan, np.ascontiguousarray(F[q]))
        fine = np.isfinite(one)
        assert np.array_equal(np.isfinite(got[q]), fine)
        assert 0 < fine.sum() and np.abs(got[q] - one)[fine].max() <= 1e-6 * np.abs(one[fine]).max()
