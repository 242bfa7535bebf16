"""Water tables at the lengths where the dose of a small plan changes its kernel, and
the longest a plan takes (GPU): one and several fluence vectors."""
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


@pytest.mark.parametrize("w_n", [768, 769, 3072])
def test_doses_with_long_water_tables(dc, oracle_mod, w_n):
    from parity_util import assert_dose_close
    p = synth.small_plan(95, n=(11, 10, 9), vox=0.3, n_beams=2, roi=1.2)
    p.comm = synth.make_commissioning(roi_radius=1.2, smooth_sigma=0.6, w_dt=0.01, w_tmax=0.01 * (w_n - 1))
    assert p.comm.water.shape[1] == w_n
    plan = dc.dc_fspb_create_from(p)
    F = np.random.default_rng(w_n).uniform(0, 1, (18, plan.n_beamlets)).astype(np.float32)
    F[0] = p.fluence
    one = [dc.dc_fspb_dose(plan, np.ascontiguousarray(f)) for f in F]
    want, amb = oracle_mod.OraclePlan(p).dose(with_amb=True)
    assert_dose_close(one[0], want, amb, label=f"w_n {w_n}")
    for k in (2, 18):
        got = dc.dc_fspb_dose_batch(plan, np.ascontiguousarray(F[:k]))
        for q in range(k):
            assert np.abs(got[q] - one[q]).max() <= 1e-6 * one[q].max()
