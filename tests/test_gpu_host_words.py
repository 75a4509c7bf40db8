"""The pinned words that tell the host of timed-out waits, shared out of pages.

A plan whose wait runs out is reported, plans beside it are not, a plan that takes
over its word starts clean, and plans whose kernels wait for nothing (vector
loads, one-frame form) need no word."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_words_belong_to_their_plans(monkeypatch):
    import paper_2203_14906_gb300 as pa
    from paper_2203_14906_gb300._native import PA_ETIMEOUT, PAError

    wl = synth.workload("cfg1", nx=64, nz=64, z1_m=10e-3)
    store, _ = synth.quantize(synth.make_frame(wl, 1)[None], "bf16")
    bf16 = pa.make_desc(wl, order_k=3, rf_dtype="bf16", compensated=1)
    f32 = pa.make_desc(wl, order_k=3)

    def run(plan, rf=store.view(np.uint16)):
        return pa.beamform_host(plan, rf, pa.PA_STAGE_ENV)

    monkeypatch.setenv("PA_ITEM_FRAMES", "1")
    before = pa.Plan(bf16, checked=True)
    loads = pa.Plan(f32, checked=True)
    assert loads.info()["tma_staging"] == 0
    rf32 = synth.make_frame(wl, 1)[None].astype(np.float32)
    ref, ref32 = run(before), run(loads, rf32)
    monkeypatch.setenv("PA_INJECT_TMA_SHORTFALL", "1")
    late = pa.Plan(bf16, checked=True)
    monkeypatch.delenv("PA_INJECT_TMA_SHORTFALL")
    with pytest.raises(PAError) as e:
        run(late)
    assert e.value.status == PA_ETIMEOUT
    assert np.array_equal(run(before), ref) and np.array_equal(run(loads, rf32), ref32)
    late.close()
    with pa.Plan(bf16, checked=True) as after:
        for _ in range(3):
            assert np.array_equal(run(after), ref)
        assert after.info()["device_error_flags"] == 0
    assert np.array_equal(run(before), ref)
    before.close()
    loads.close()
