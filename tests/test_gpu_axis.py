"""The axis stencil's taps (GPU) where they change their form: voxels whose taps
lie inside the grid, cross its border or all leave it, on grids of one, two and
odd numbers of voxels per side and away from the origin, against the FP64 oracle."""
import numpy as np
import pytest

from paper_1103_1164_gb300 import synth
from parity_util import assert_dose_close

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


@pytest.mark.parametrize("n", [(1, 9, 7), (9, 1, 6), (6, 9, 1), (2, 13, 2), (5, 5, 5), (23, 17, 19)])
def test_axis_dose_at_the_border(dc, oracle_mod, n):
    p = synth.small_plan(60, n=n, vox=0.35, n_beams=3, field=3.0, couch=True, phantom="water")
    p.rho = np.random.default_rng(61).uniform(0.3, 1.7, p.rho.shape).astype(np.float32)
    plan = dc.dc_fspb_create_from(p, lateral_mode=dc.DC_LATERAL_AXIS)
    got = dc.dc_fspb_dose(plan, p.fluence)
    want, amb = oracle_mod.OraclePlan(p, lateral_mode=1).dose(with_amb=True)
    assert_dose_close(got, want, amb, label=f"axis border {n}")
