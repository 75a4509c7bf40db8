"""Every variant of every form of the fused kernel, and which form ran.

The forms (one frame per work item, two, one and two pixels per thread) give
the same bits, so a comparison says nothing if a plan quietly keeps another form:
each case here asserts the form that its launch runs (pa_plan_form).  Blocks of 4
and 8 warps (4 and 8 columns a pitch), where compensated plans have every form;
all orders, apodisation, Kahan sums, samples and tables; release and checked
build; waits that run out in each form.  The tests of the one-frame kernel's
staging, lane groups and tensor-memory sums run again with that form asked for:
small launches run another one by themselves.
"""

import itertools

import numpy as np
import pytest

import synth
import test_gpu_failure as failure
import test_gpu_parity as parity

pytestmark = pytest.mark.gpu

ONE, TWO, FINE1, FINE2 = 1, 2, 3, 4


def _wl(m, **kw):
    n = 40
    wl = synth.workload("cfg1", n_elem=n, n_samples=402, nx=n * m, nz=70, z0_m=0.3e-3, z1_m=12e-3, **kw)
    half = n * wl["pitch_m"] / 2
    wl["x0_m"], wl["x1_m"] = -half, half
    return wl


def _has(form, k, comp, table):
    """Whether the form has a kernel for these sums."""
    if form == TWO:
        return k <= 5
    if form == FINE1:
        return not (comp and table == "full" and k == 8)
    return form == ONE or (not comp and k <= 5 and (table == "full" or k >= 3))


def _run(wl, k, form, rf, frames, monkeypatch, dtype="f32", checked=False):
    import torch

    import paper_2203_14906_gb300 as pa

    monkeypatch.setenv("PA_ITEM_FRAMES", str(form))
    desc = pa.make_desc(wl, order_k=k, outputs=7, rf_dtype=dtype, max_batch=frames)
    with pa.Plan(desc, checked=checked) as plan:
        assert plan.form(frames) == form, (k, form)
        out = pa.beamform(plan, rf, pa.PA_STAGE_RAW)
        torch.cuda.synchronize()
        assert plan.info()["device_error_flags"] == 0
    return out


def _frames(wl, frames, dtype="f32"):
    import torch

    rf = np.stack([synth.make_frame(wl, 60 + f) for f in range(frames)])
    store, _ = synth.quantize(rf, dtype)
    if dtype == "bf16":
        return torch.from_numpy(store.view(np.int16)).cuda().view(torch.bfloat16)
    return torch.from_numpy(store).cuda()


@pytest.mark.parametrize("m", [4, 8])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 5, 6, 7, 8])
def test_every_variant_runs_and_has_the_one_frame_bits(m, k, monkeypatch):
    import torch

    for f_number, comp, interp, table in itertools.product((0.0, 1.4), (0, 1), ("linear", "nearest"),
                                                           ("lattice", "full")):
        if m == 8 and table == "full":
            continue  # (full-table plans choose their own column stride)
        wl = _wl(m, f_number=f_number, interp=interp, delay_table=table, compensated=comp)
        rf = _frames(wl, 3)
        ref = _run(wl, k, ONE, rf, 3, monkeypatch)
        assert float(ref.abs().max()) > 0
        for form in (TWO, FINE1, FINE2):
            if not _has(form, k, comp, table):
                continue
            out = _run(wl, k, form, rf, 3, monkeypatch)
            assert torch.equal(out, ref), (form, f_number, comp, interp, table)


@pytest.mark.parametrize("form", [ONE, TWO, FINE1, FINE2])
@pytest.mark.parametrize("k,m,comp,f_number,interp,table,dtype", [
    (3, 4, 0, 0.0, "linear", "lattice", "f32"), (3, 4, 1, 0.0, "linear", "lattice", "bf16"),
    (4, 4, 0, 1.4, "nearest", "lattice", "bf16"),
    (5, 8, 1, 0.0, "nearest", "lattice", "f32"), (2, 4, 1, 1.4, "linear", "lattice", "f16"),
    (2, 4, 0, 1.4, "nearest", "full", "f32"), (4, 4, 1, 1.4, "linear", "full", "bf16")])
def test_checked_build_of_every_form(form, k, m, comp, f_number, interp, table, dtype, monkeypatch):
    if not _has(form, k, comp, table):
        pytest.skip("no such kernel")
    wl = _wl(m, f_number=f_number, interp=interp, delay_table=table, compensated=comp)
    _run(wl, k, form, _frames(wl, 3, dtype), 3, monkeypatch, dtype=dtype, checked=True)


@pytest.mark.parametrize("form", [ONE, TWO, FINE1, FINE2])
def test_a_wait_that_runs_out_is_reported(form, monkeypatch):
    """Every chunk expects 16 bytes more than its copies bring (checked build): each
    block gives up after about a second, and the host path says so."""
    import paper_2203_14906_gb300 as pa
    from paper_2203_14906_gb300._native import PA_ETIMEOUT, PAError

    wl = synth.workload("cfg1", nx=128, nz=64, z1_m=10e-3)  # 2 columns a pitch: 4 warps
    store, _ = synth.quantize(np.stack([synth.make_frame(wl, s) for s in (1, 2)]), "bf16")
    desc = pa.make_desc(wl, order_k=3, rf_dtype="bf16", compensated=int(form != FINE2), max_batch=2)
    monkeypatch.setenv("PA_ITEM_FRAMES", str(form))
    for shortfall in (True, False):
        if shortfall:
            monkeypatch.setenv("PA_INJECT_TMA_SHORTFALL", "1")
        else:
            monkeypatch.delenv("PA_INJECT_TMA_SHORTFALL")
        with pa.Plan(desc, checked=True) as plan:
            plan.set_host_schedule(2, pa.PA_STAGE_LOG, [2])
            assert plan.form(2) == form and plan.info()["tma_staging"] == 1
            if shortfall:
                with pytest.raises(PAError) as e:
                    pa.beamform_host(plan, store.view(np.uint16), pa.PA_STAGE_LOG)
                assert e.value.status == PA_ETIMEOUT
                assert plan.info()["device_error_flags"] & 8
            else:
                out = pa.beamform_host(plan, store.view(np.uint16), pa.PA_STAGE_LOG)
                assert plan.info()["device_error_flags"] == 0
                assert np.isfinite(out).all() and out.max() == 0.0


def test_the_one_frame_kernel_by_itself(monkeypatch):
    monkeypatch.setenv("PA_ITEM_FRAMES", "1")
    for dtype in ("f32", "bf16", "f16"):
        with monkeypatch.context() as mp:
            parity.test_tma_and_load_staging_agree(dtype, mp)
    for test in (parity.test_lane_groups_keep_bits, parity.test_lane_groups_with_tmem_sums):
        with monkeypatch.context() as mp:
            test(mp)
    parity.test_checked_build_raises_no_bounds_flags()
    parity.test_full_table_checked_build()


def test_the_one_frame_kernels_timed_out_wait(monkeypatch):
    monkeypatch.setenv("PA_ITEM_FRAMES", "1")
    with monkeypatch.context() as mp:
        failure.test_bounded_wait_reports_timeout_on_the_host_path(mp)
    with monkeypatch.context() as mp:
        failure.test_server_completes_a_timed_out_batch_with_etimeout(mp)


def test_forms_outside_the_plans_launches_are_refused():
    import paper_2203_14906_gb300 as pa
    from paper_2203_14906_gb300._native import PA_EINVAL, PAError

    with pa.Plan(pa.make_desc(_wl(4), order_k=3, max_batch=2)) as plan:
        assert plan.form(1) in (1, 3) and plan.form(2) in (1, 2, 3)
        for n in (0, 3):
            with pytest.raises(PAError) as e:
                plan.form(n)
            assert e.value.status == PA_EINVAL
