"""The backward pass's sums (GPU) by identities that hold for every table: the
dose is linear in omega_1, omega_2 = f_omega (omega^w + omega^corr), so the
gradients times the tables give back the weighted dose.  Slabs (a warp's lanes
share their bins), random densities (they do not), tables that end inside the
body and densities outside the functions' domain."""
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


@pytest.mark.parametrize("w_dt,w_tmax", [(0.125, 80.0), (0.4, 2.0), (3.0, 3.0)])
@pytest.mark.parametrize("body", ["water", "slab", "random"])
def test_gradients_reproduce_the_dose(dc, body, w_dt, w_tmax):
    rng = np.random.default_rng(90)
    p = synth.small_plan(91, n=(17, 15, 13), vox=0.45, n_beams=2, field=3.0, roi=1.8, couch=True,
                         phantom="slab" if body == "slab" else "water")
    if body == "random":
        p.rho = rng.uniform(0.05, 2.4, p.rho.shape).astype(np.float32)
    p.comm = synth.make_commissioning(roi_radius=1.8, smooth_sigma=0.3, w_dt=w_dt, w_tmax=w_tmax)
    plan = dc.dc_fspb_create_from(p)
    cm = p.comm
    wv = rng.uniform(0, 1, plan.n_voxels).astype(np.float32)
    wv[::5] = 0
    gw, gd, gc = dc.dc_fspb_dose_vjp(plan, p.fluence, wv, cm.water.shape[1], cm.dens.shape[1])
    want = float(dc.dc_fspb_dose(plan, p.fluence).reshape(-1).astype(np.float64) @ wv)
    assert want > 0
    by_water = float((gw[2:4].astype(np.float64) * cm.water[2:4]).sum() + gc.astype(np.float64).sum())
    by_density = float((gd[2:4].astype(np.float64) * cm.dens[2:4]).sum())
    # FP32 pair values of two forms (a few 1e-6 each) and sums of positive terms in FP32
    assert abs(by_water - want) <= 1e-4 * want
    assert abs(by_density - want) <= 1e-4 * want
