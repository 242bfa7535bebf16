"""The backward pass (GPU) with one, two and four work items per unit, which it
chooses by the number of units and the beamlets of a window: the dose is linear in
omega_1, omega_2 = f_omega (omega^w + omega^corr), so the gradients times the
tables give back the weighted dose, whichever form computes them."""
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


# 8,192, 24,576 and 73,728 units of 41 beamlets, 24,576 of 127
@pytest.mark.parametrize("n_beams,roi", [(1, 1.8), (3, 1.8), (9, 1.8), (3, 3.18)])
def test_gradients_reproduce_the_dose(dc, n_beams, roi):
    p = synth.small_plan(93, n=(64, 64, 64), vox=0.3, n_beams=n_beams, field=4.0, roi=roi, couch=True)
    plan = dc.dc_fspb_create_from(p)
    cm = p.comm
    wv = np.random.default_rng(94).uniform(0, 1, plan.n_voxels).astype(np.float32)
    gw, gd, gc = dc.dc_fspb_dose_vjp(plan, p.fluence, wv, cm.water.shape[1], cm.dens.shape[1])
    want = float(dc.dc_fspb_dose(plan, p.fluence).reshape(-1).astype(np.float64) @ wv)
    assert want > 0
    by_water = float((gw[2:4].astype(np.float64) * cm.water[2:4]).sum() + gc.astype(np.float64).sum())
    by_density = float((gd[2:4].astype(np.float64) * cm.dens[2:4]).sum())
    # FP32 pair values of two forms (a few 1e-6 each) and sums of positive terms in FP32
    assert abs(by_water - want) <= 1e-4 * want
    assert abs(by_density - want) <= 1e-4 * want
