"""The pair counts and the matrix pattern of the passes that settle beamlets for a
warp's whole box of voxels (GPU), on the ragged and degenerate cases of
test_gpu_windows, against the FP64 oracle's own traversal: each sampled row holds
every pair the oracle includes outside its rounding margins and none it excludes,
its columns ascend, and its length is the counted one."""
import numpy as np
import pytest

from test_gpu_windows import CASES, _plan

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


@pytest.mark.parametrize("counted_by_the_dose", [False, True])
@pytest.mark.parametrize("air", [False, True])
@pytest.mark.parametrize("j", range(len(CASES)))
def test_rows_hold_the_oracles_pairs(dc, oracle_mod, j, air, counted_by_the_dose):
    p = _plan(j, air)
    plan = dc.dc_fspb_create_from(p)
    if counted_by_the_dose:
        dc.dc_fspb_dose(plan, p.fluence)
    pairs = dc.dc_fspb_pair_count(plan)
    rowptr, cols, _ = dc.dc_fspb_dose_matrix(plan)
    assert rowptr[0] == 0 and rowptr[-1] == pairs > 0
    op = oracle_mod.OraclePlan(p)
    vox = np.unique(np.random.default_rng(j).integers(0, op.V, 600))
    o_ptr, o_cols, _, o_flags = op.matrix(vox)
    for r, v in enumerate(vox):
        got = cols[rowptr[v]:rowptr[v + 1]]
        sl = slice(o_ptr[r], o_ptr[r + 1])
        oc, of = o_cols[sl], o_flags[sl]
        must = oc[((of & 1) != 0) & ((of & 2) == 0)]
        assert np.all(np.diff(got) > 0), v
        assert np.isin(must, got).all() and np.isin(got, oc).all(), v
