"""Several fluence vectors (GPU) on plans of few work units, which two warps share,
and of many: k vectors give the doses of the same vectors among 64, which take
another form, to the bit; k up to the widths 16 and 32, windows of a few to several
hundred beamlets, merged and general tables, non-finite fluences."""
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


def _plans():
    yield synth.small_plan(580, n=(21, 19, 17), vox=0.25, n_beams=3, field=3.0, roi=0.4)
    yield synth.small_plan(581, n=(13, 23, 12), vox=0.3, n_beams=2, field=5.0, beamlet=0.25, roi=3.0, couch=True)
    yield synth.small_plan(582, n=(24, 24, 14), vox=0.25, n_beams=1, field=9.0, beamlet=0.25, roi=2.0)
    yield synth.config2(0.375)   # 23,328 units


@pytest.mark.parametrize("j", range(4))
def test_same_bits_as_among_64_vectors(dc, j):
    plan = dc.dc_fspb_create_from(list(_plans())[j])
    F = np.random.default_rng(j).uniform(0, 1, (64, plan.n_beamlets)).astype(np.float32)
    for bad in (False, True):
        if bad:
            F[0, 3], F[1, plan.n_beamlets // 2], F[1, plan.n_beamlets - 1] = np.inf, np.nan, -np.inf
        all64 = dc.dc_fspb_dose_batch(plan, F)
        assert np.nanmax(np.abs(all64[2:])) > 0
        for k in (2, 3, 15, 16, 17, 31, 32):
            got = dc.dc_fspb_dose_batch(plan, np.ascontiguousarray(F[:k]))
            assert np.array_equal(got, all64[:k], equal_nan=True), k
