"""Sums over beams (GPU): the SpMM's for every group width and both load forms
(even and odd numbers of vectors, an output off an 8-byte boundary), and the
fluence batch's, with more beams than are loaded at a time."""
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


@pytest.mark.parametrize("n_beams", [2, 8, 11, 17])
def test_spmm_columns_do_not_depend_on_their_number(dc, n_beams):
    import torch
    plan = dc.dc_fspb_create_from(synth.small_plan(70 + n_beams, n=(15, 13, 10), vox=0.3, n_beams=n_beams, field=2.0,
                                                   beamlet=0.5, roi=1.5, couch=True))
    dc.dc_fspb_spmm_prepare(plan)
    F = torch.rand(plan.n_beamlets, 64, device="cuda", generator=torch.Generator("cuda").manual_seed(n_beams))
    full = torch.empty(plan.n_voxels, 64, device="cuda")
    dc.dc_fspb_spmm(plan, F, full)
    assert float(full.abs().max()) > 0
    for k in (1, 2, 7, 15, 16, 17, 31, 32, 33, 63):
        for off in (0, 1):
            Y = torch.empty(plan.n_voxels * k + 1, device="cuda")[off:off + plan.n_voxels * k].view(plan.n_voxels, k)
            dc.dc_fspb_spmm(plan, F[:, :k].contiguous(), Y)
            assert torch.equal(Y, full[:, :k]), (k, off)


@pytest.mark.parametrize("n_beams", [1, 5, 6, 13])
def test_batch_sums_in_beam_order(dc, n_beams):
    plan = dc.dc_fspb_create_from(synth.small_plan(80 + n_beams, n=(13, 11, 9), vox=0.35, n_beams=n_beams, roi=1.2))
    F = np.random.default_rng(n_beams).uniform(0, 1, (20, plan.n_beamlets)).astype(np.float32)
    one = [dc.dc_fspb_dose(plan, np.ascontiguousarray(f)) for f in F]
    for k in (2, 4, 5, 8, 9, 20):
        got = dc.dc_fspb_dose_batch(plan, np.ascontiguousarray(F[:k]))
        for q in range(k):
            assert np.abs(got[q] - one[q]).max() <= 1e-6 * one[q].max()
