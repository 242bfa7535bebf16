"""Calls on a live plan after another call has run out of device memory (GPU): the
allocation fails in the CUDA runtime itself, which then holds an error of its own
until it is taken; doses, with other fluences than before, and the matrix pattern
must be those of a plan that saw no failure, and no call may report the other's
error.  Plans of few units (a CTA per unit) and of many (a warp per unit)."""
import ctypes as C

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


def _gamma_of_2_40_voxels(dc):
    # 4 TiB for the device copy of the first dose: refused before any host element is read
    x = np.zeros(1, np.float32)
    g = dc.dc_grid(4096, 16384, 16384, 0.3, 0.3, 0.3, 0.0, 0.0, 0.0)
    return dc.load().dc_gamma_index(x.ctypes.data, x.ctypes.data, C.byref(g), 3.0, 0.3, 0.6, None, None,
                                    C.c_void_p(0), 0)


def _gradient_of_2_31_samples(dc):
    # 412 GB for the device copy of the samples: refused before any host element is read
    net = dc.Mlp(np.zeros(dc.MLP_PARAMS, np.float32))
    x = np.zeros(dc.MLP_PARAMS, np.float32)
    return dc.load().dc_mlp_gradient(net.handle, x.ctypes.data, x.ctypes.data, 2**31 - 1, x.ctypes.data, None, 0)


def _calls(dc, p, plan):
    """Calls of a live plan, in an order in which each next one depends on the ones before."""
    rng = np.random.default_rng(7)
    f = rng.uniform(0, 1, (20, plan.n_beamlets)).astype(np.float32)
    yield "dose", lambda: dc.dc_fspb_dose(plan, f[0])
    yield "dose of another fluence", lambda: dc.dc_fspb_dose(plan, f[1])
    yield "pair count", lambda: dc.dc_fspb_pair_count(plan)
    yield "several vectors", lambda: dc.dc_fspb_dose_batch(plan, f)
    yield "density", lambda: dc.dc_fspb_set_density(plan, np.float32(0.9) * p.rho)
    yield "dose of the density", lambda: dc.dc_fspb_dose(plan, f[2])
    yield "axis form", lambda: dc.dc_fspb_set_lateral_mode(plan, dc.DC_LATERAL_AXIS)
    yield "its dose", lambda: dc.dc_fspb_dose(plan, f[3])
    yield "pair count of the density", lambda: dc.dc_fspb_pair_count(plan)
    yield "tiles", lambda: dc.dc_fspb_spmm_prepare(plan)
    yield "product", lambda: dc.dc_fspb_spmm(plan, f[:5].T.copy())


@pytest.mark.parametrize("fail", [_gamma_of_2_40_voxels, _gradient_of_2_31_samples])
@pytest.mark.parametrize("many_units", [False, True])
def test_calls_after_a_failed_allocation(dc, many_units, fail):
    p = synth.config2(0.375) if many_units else synth.small_plan(511, n=(15, 16, 11), vox=0.25, n_beams=3, roi=2.0)
    fresh, live = dc.dc_fspb_create_from(p), dc.dc_fspb_create_from(p)
    want = [call() for _, call in _calls(dc, p, fresh)]
    reported, wrong = [], []
    for (name, call), w in zip(_calls(dc, p, live), want):
        assert fail(dc) == dc.DC_ENOMEM
        try:
            got = call()
        except dc.DcError as e:
            reported.append((name, str(e)))
            continue
        if w is not None and not np.array_equal(got, w):
            wrong.append(name)
    assert not wrong and not reported


def test_batch_after_a_plan_lost_its_partial_doses(dc, monkeypatch):
    # 64 vectors want a larger buffer of partial doses, whose allocation fails: the
    # batch's captured graphs must not use the one that was freed for it
    plans = [synth.small_plan(520 + j, n=(15, 16, 11), vox=0.25, n_beams=3, roi=2.0) for j in range(2)]
    live = [dc.dc_fspb_create_from(p) for p in plans]
    fluences = [p.fluence for p in plans]
    want = [dc.dc_fspb_dose(dc.dc_fspb_create_from(p), p.fluence).reshape(-1) for p in plans]
    for variant in range(3):
        batch = dc.dc_fspb_batch_create(live)
        dc.dc_fspb_batch_set_variant(batch, variant)
        for fail_again in (False, True):
            for density in (False, True):
                for got, w in zip(dc.dc_fspb_batch_dose(batch, fluences, density=density), want):
                    assert np.array_equal(got.reshape(-1), w)
            # plan creation leaves room for one vector, the batch for no more
            F = np.ones((64, live[0].n_beamlets), np.float32)
            monkeypatch.setenv("DC_FSPB_FAIL_ALLOC_AT", "1")
            with pytest.raises(dc.DcError) as ei:
                dc.dc_fspb_dose_batch(live[0], F)
            assert ei.value.status == dc.DC_ENOMEM
            if fail_again:   # no memory for the batch either: an error, no launch
                monkeypatch.setenv("DC_FSPB_FAIL_ALLOC_AT", "01")
                with pytest.raises(dc.DcError) as ei:
                    dc.dc_fspb_batch_dose(batch, fluences)
                assert ei.value.status == dc.DC_ENOMEM
            monkeypatch.delenv("DC_FSPB_FAIL_ALLOC_AT")
