"""The passes that settle beamlets for a warp's whole box of voxels at once
(GPU): the pair counts of the count pass against those the dose pass records
pair by pair, and the SpMM's tiles, whose patches the mark pass finds the same
way, against the CSR matrix's product, over ROI radii from under a voxel to
beyond the field, rectangular beamlets, rotated beams, bodies that end inside
the grid and grids of ragged and degenerate size."""
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


CASES = [dict(n=(33, 29, 21), vox=0.25, n_beams=3, field=4.0, roi=5.0),
         dict(n=(33, 29, 21), vox=0.25, n_beams=2, field=6.0, roi=1.0),
         dict(n=(20, 31, 17), vox=0.3, n_beams=2, field=3.0, roi=0.2),
         dict(n=(24, 24, 24), vox=0.3, n_beams=2, field=8.0, beamlet=0.2, beamlet_y=0.5, roi=2.0, couch=True),
         dict(n=(40, 9, 33), vox=0.25, n_beams=5, field=5.0, beamlet=0.25, roi=3.0, couch=True, phantom="water"),
         dict(n=(1, 37, 5), vox=0.5, n_beams=2, field=2.0, roi=2.0, phantom="water"),
         dict(n=(9, 70, 9), vox=0.25, n_beams=1, field=12.0, beamlet=0.25, roi=4.0, phantom="slab")]


def _plan(j, air):
    p = synth.small_plan(900 + j, **CASES[j])
    if air:   # a body that ends inside the grid, with a cavity: depth decides there
        X = np.indices(p.rho.shape).astype(np.float32)
        c = [(s - 1) / 2 for s in p.rho.shape]
        r = sum(((X[a] - c[a]) / max(0.45 * p.rho.shape[a], 1.0)) ** 2 for a in range(3))
        p.rho = np.where((r <= 1.0) & (r >= 0.05), p.rho, np.float32(0.001)).astype(np.float32)
    return p


@pytest.mark.parametrize("air", [False, True])
@pytest.mark.parametrize("j", range(len(CASES)))
def test_counts_equal_the_dose_pass_counts(dc, j, air):
    p = _plan(j, air)
    a, b = dc.dc_fspb_create_from(p), dc.dc_fspb_create_from(p)
    na = dc.dc_fspb_pair_count(a)          # count pass
    dc.dc_fspb_dose(b, p.fluence)          # records the counts
    assert na == dc.dc_fspb_pair_count(b)
    ra, ca, va = dc.dc_fspb_dose_matrix(a)
    rb, cb, vb = dc.dc_fspb_dose_matrix(b)
    assert np.array_equal(ra, rb) and np.array_equal(ca, cb) and np.array_equal(va, vb)


@pytest.mark.parametrize("air", [False, True])
@pytest.mark.parametrize("j", range(len(CASES)))
def test_tiles_hold_every_pair(dc, j, air):
    p = _plan(j, air)
    plan = dc.dc_fspb_create_from(p)
    dc.dc_fspb_spmm_prepare(plan)
    F = np.random.default_rng(j).uniform(0, 1, (plan.n_beamlets, 3)).astype(np.float32)
    got = dc.dc_fspb_spmm(plan, F)
    rp, cols, vals = dc.dc_fspb_dose_matrix(plan, dc.DC_BF16)
    M = (vals.astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    u = F.view(np.uint32).astype(np.uint64)
    Fb = (((u + 0x7fff + ((u >> 16) & 1)) >> 16) << 16).astype(np.uint32).view(np.float32).astype(np.float64)
    want = np.zeros((plan.n_voxels, 3))
    np.add.at(want, np.repeat(np.arange(plan.n_voxels), np.diff(rp)), M[:, None] * Fb[cols])
    # FP32 accumulation of at most a few thousand products
    assert np.all(np.abs(got - want) <= 1e-5 * np.abs(want).max(0) + 1e-9)
