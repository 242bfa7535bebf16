"""Gamma calls (GPU) that share the device's scratch: more calls at once than it
has slots, search spheres beyond a slot's offsets, and a call after a refused one."""
import threading

import numpy as np
import pytest

from oracle import gamma as og
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


def _doses(shape, seed):
    rng = np.random.default_rng(seed)
    ref = rng.uniform(0.2, 1.0, shape).astype(np.float32)
    return ref, (ref * rng.uniform(0.95, 1.05, shape)).astype(np.float32)


def test_many_calls_at_once(dc):
    import torch
    jobs = []
    for t in range(9):
        shape = (5 + 7 * t, 33 - t, 20 + 3 * t)
        ref, ev = (torch.from_numpy(a).cuda() for a in _doses(shape, t))
        jobs.append((ref, ev, synth.centred_grid(shape[2], shape[1], shape[0], 0.2), 0.3 + 0.1 * t))
    alone = [dc.dc_gamma_index(r, e, g, search=s) for r, e, g, s in jobs]
    torch.cuda.synchronize()
    got, bad = [None] * len(jobs), []

    def work(i):
        r, e, g, s = jobs[i]
        try:
            st = torch.cuda.Stream()
            out = torch.full_like(r, -1.0)
            torch.cuda.synchronize()
            for _ in range(8):
                got[i] = dc.dc_gamma_index(r, e, g, search=s, gamma=out, stream=st.cuda_stream)
                if got[i][1] != alone[i][1]:
                    bad.append(i)
        except Exception as x:   # noqa: BLE001
            bad.append((i, x))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
    for (g0, _), (g1, _) in zip(alone, got):
        assert torch.equal(g0, g1)


@pytest.mark.parametrize("search", [0.97, 1.2])   # 3,863 and 7,153 offsets on this grid
def test_offsets_around_a_slot(dc, search):
    ref, ev = _doses((9, 11, 14), 3)
    ev = np.ascontiguousarray(ev * np.float32(1.3))   # far offsets decide in places
    g = synth.centred_grid(14, 11, 9, 0.1)
    gamma, st = dc.dc_gamma_index(ref, ev, g, pct=1.0, dta=0.3, search=search)
    want = og.gamma_index(ref, ev, (0.1, 0.1, 0.1), pct=1.0, dta=0.3, radius=search)
    # FP32 distance and dose terms, as the bound for the gamma kernel elsewhere
    assert np.abs(gamma - want).max() < 2e-5 + 1e-5 * want.max()
    assert st["n50"] == int((ref >= 0.5 * ref.max()).sum())


def test_call_after_a_refused_one(dc):
    ref, ev = _doses((6, 7, 8), 4)
    g = synth.centred_grid(8, 7, 6, 0.25)
    first = dc.dc_gamma_index(ref, ev, g)
    out = np.full(ref.shape, 7.0, np.float32)
    with pytest.raises(Exception, match="zero everywhere"):
        dc.dc_gamma_index(np.zeros_like(ref), ev, g, gamma=out)
    assert (out == 7.0).all()
    again = dc.dc_gamma_index(ref, ev, g)
    assert np.array_equal(first[0], again[0]) and first[1] == again[1]
