"""The density steps (GPU): the smoothed density on grids whose sides are not
multiples of a run of outputs, or shorter than the kernel's reach, against the
FP64 oracle, and a plan that gets a new density against one created with it."""
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


@pytest.mark.parametrize("sigma", [0.0, 0.2, 1.1])
@pytest.mark.parametrize("n", [(1, 6, 9), (5, 1, 4), (7, 3, 1), (13, 10, 11), (2, 33, 18)])
def test_smoothed_density(dc, oracle_mod, n, sigma):
    p = synth.small_plan(40, n=n, vox=0.4, phantom="water")
    p.rho = np.random.default_rng(41).uniform(0, 2, p.rho.shape).astype(np.float32)
    p.comm.smooth_sigma = sigma
    want = oracle_mod.OraclePlan(p).smoothed()
    got = dc.dc_fspb_get_smoothed(dc.dc_fspb_create_from(p))
    # three axes of at most 19 taps: each tap's weight, product and sum rounds once
    assert np.abs(got - want).max() <= 3 * (19 + 2) * 2.0 ** -24 * 2.0
    if sigma == 0:
        assert np.array_equal(got, p.rho)


@pytest.mark.parametrize("merged", [False, True])
def test_new_density_equals_a_new_plan(dc, merged):
    p = synth.small_plan(42, n=(19, 14, 11), vox=0.3, n_beams=3, field=3.0, couch=True)
    if merged:   # water tables on the beamlets' depth grid
        p.comm.w_dt = 0.15
    old = dc.dc_fspb_create_from(p)
    rho = p.rho.copy()
    rho[:, :5] = 0.001   # another body: entry, exit and table lengths change
    dc.dc_fspb_set_density(old, rho)
    p.rho = rho
    new = dc.dc_fspb_create_from(p)
    assert np.array_equal(dc.dc_fspb_get_beamlets(old).view(np.uint32), dc.dc_fspb_get_beamlets(new).view(np.uint32))
    for i in range(0, new.n_beamlets, 7):
        for a, b in zip(dc.dc_fspb_get_tables(old, i), dc.dc_fspb_get_tables(new, i)):
            assert np.array_equal(a, b)
    ra, ca, va = dc.dc_fspb_dose_matrix(old)
    rb, cb, vb = dc.dc_fspb_dose_matrix(new)
    assert np.array_equal(ra, rb) and np.array_equal(ca, cb) and np.array_equal(va, vb)
