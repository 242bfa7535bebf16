"""The SpMM's sum over beams (GPU) in its three forms, up to 16, up to 32 and more
columns, on plans of more beams than a warp has lanes: a column's sum does not
depend on the number of columns, and is the CSR matrix's product."""
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


@pytest.mark.parametrize("n_beams", [3, 32, 33, 64])
def test_columns_of_many_beams(dc, n_beams):
    plan = dc.dc_fspb_create_from(synth.small_plan(590 + n_beams, n=(12, 11, 9), vox=0.35, n_beams=n_beams, field=1.5,
                                                   beamlet=0.5, roi=1.2, couch=True))
    dc.dc_fspb_spmm_prepare(plan)
    F = np.random.default_rng(n_beams).uniform(0, 1, (plan.n_beamlets, 64)).astype(np.float32)
    full = dc.dc_fspb_spmm(plan, F)
    rp, cols, vals = dc.dc_fspb_dose_matrix(plan, dc.DC_BF16)
    M = (vals.astype(np.uint32) << 16).view(np.float32).astype(np.float64)
    u = F.view(np.uint32).astype(np.uint64)
    Fb = (((u + 0x7fff + ((u >> 16) & 1)) >> 16) << 16).astype(np.uint32).view(np.float32).astype(np.float64)
    want = np.zeros((plan.n_voxels, 64))
    np.add.at(want, np.repeat(np.arange(plan.n_voxels), np.diff(rp)), M[:, None] * Fb[cols])
    # FP32 accumulation of at most a few hundred products per beam
    assert want.max() > 0 and np.all(np.abs(full - want) <= 1e-5 * np.abs(want).max(0))
    for k in (5, 16, 17, 32, 33, 50, 63):
        assert np.array_equal(dc.dc_fspb_spmm(plan, np.ascontiguousarray(F[:, :k])), full[:, :k]), k
