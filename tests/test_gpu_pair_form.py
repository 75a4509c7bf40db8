"""The two-frame and fine-grained forms of the fused kernel give the one-frame
form's bits.

PA_ITEM_FRAMES picks the form (1: one frame per work item, 2: two, 3: one pixel
per thread); each pixel's arithmetic is the same in both, so
images are compared bit by bit over the forms the kernel is built for: orders
1-5, linear and nearest samples, plain and compensated sums, apodisation,
lattice and full delay tables, the RF types, even and odd frame counts, records
with rows off 16-byte boundaries, and records so short that whole windows lie
past their end.  One frame of each is held to the oracle (1e-4 of the peak).
"""

import numpy as np
import pytest

import synth
from gpu_util import assert_parity, compare, oracle_frames, run_gpu

pytestmark = pytest.mark.gpu

CASES = [
    # k, dtype, comp, f_number, interp, table, Ns, frames
    (1, "f32", 0, 0.0, "linear", "auto", 512, 2),
    (2, "f32", 0, 0.0, "nearest", "auto", 333, 3),
    (2, "bf16", 1, 1.5, "nearest", "auto", 512, 4),
    (2, "f16", 1, 0.0, "linear", "full", 331, 5),
    (3, "f32", 0, 0.0, "linear", "auto", 513, 7),
    (3, "f32", 0, 0.0, "nearest", "full", 512, 2),
    (3, "bf16", 1, 0.0, "linear", "auto", 512, 6),
    (3, "f32", 1, 1.3, "nearest", "auto", 181, 3),
    (4, "f32", 0, 0.0, "nearest", "auto", 334, 2),
    (4, "bf16", 1, 1.5, "linear", "auto", 512, 3),
    (4, "f32", 0, 1.2, "linear", "full", 257, 4),
    (5, "f16", 0, 0.0, "linear", "auto", 335, 2),
    (5, "f32", 1, 0.0, "nearest", "auto", 512, 9),
    (5, "f32", 0, 2.0, "linear", "auto", 512, 2),
]


def _wl(ns, f_number, interp, table, **kw):
    wl = synth.workload("cfg1", n_elem=45, n_samples=ns, nx=150, nz=70, z0_m=0.4e-3, z1_m=11e-3,
                        f_number=f_number, interp=interp, delay_table=table, **kw)
    wl["x0_m"], wl["x1_m"] = -45 * 0.15e-3 + 0.6e-3, -45 * 0.15e-3 + 0.6e-3 + 150 * 0.1e-3
    return wl


@pytest.mark.parametrize("k,dtype,comp,f_number,interp,table,ns,frames", CASES)
def test_bits_of_the_one_frame_form(k, dtype, comp, f_number, interp, table, ns, frames,
                                    monkeypatch):
    wl = _wl(ns, f_number, interp, table)
    rf = np.stack([synth.make_frame(wl, 50 + f) for f in range(frames)])
    outs = {}
    for form in ("1", "2", "3"):
        monkeypatch.setenv("PA_ITEM_FRAMES", form)
        outs[form], info, deq = run_gpu(wl, rf, k, rf_dtype=dtype, compensated=comp)
        assert info["device_error_flags"] == 0
    assert np.array_equal(outs["1"], outs["2"]) and np.array_equal(outs["1"], outs["3"])
    last = frames - 1
    refs = oracle_frames(wl, deq[last:], k)
    assert_parity(compare(outs["2"][last:], refs), 1e-4, what=f"k={k} {interp} {table}")


def test_two_pixels_a_thread_and_high_orders():
    """Launches between the lines of the plan's own choice: two pixels a thread
    (compensated, 1200-2400 warps) and orders above 5 at one pixel."""
    wl = synth.workload("cfg1", n_elem=64, nx=256, nz=256, z1_m=20e-3)  # 512 warps a frame
    for k, frames, dtype, comp, interp in ((3, 4, "bf16", 1, "linear"), (5, 3, "f32", 1, "nearest"),
                                           (7, 1, "f32", 0, "linear"), (8, 2, "bf16", 1, "linear")):
        w = dict(wl, interp=interp)
        rf = np.stack([synth.make_frame(w, 80 + f) for f in range(frames)])
        mp = pytest.MonkeyPatch()
        out, info, _ = run_gpu(w, rf, k, rf_dtype=dtype, compensated=comp)
        mp.setenv("PA_ITEM_FRAMES", "1")
        ref, _, _ = run_gpu(w, rf, k, rf_dtype=dtype, compensated=comp)
        mp.undo()
        assert info["device_error_flags"] == 0 and np.array_equal(out, ref), (k, frames)


@pytest.mark.parametrize("form", ["2", "3"])
def test_checked_build_sees_no_access_out_of_range(form, monkeypatch):
    monkeypatch.setenv("PA_ITEM_FRAMES", form)
    for k, dtype, comp, f_number, interp, table, ns, frames in CASES[::3]:
        wl = _wl(ns, f_number, interp, table)
        rf = np.stack([synth.make_frame(wl, 50 + f) for f in range(frames)])
        _, info, _ = run_gpu(wl, rf, k, rf_dtype=dtype, compensated=comp, checked=True)
        assert info["device_error_flags"] == 0, (k, interp, table)


def test_more_frames_than_one_round_of_slots(monkeypatch):
    """140 frames of 96 x 4096 samples need more prepared slots than a launch
    holds at once, so it runs in rounds; every frame has the bits it has alone."""
    wl = synth.workload("cfg1", n_elem=96, n_samples=4096, nx=48, nz=64, z1_m=20e-3)
    one = [synth.make_frame(wl, 70 + f) for f in range(3)]
    rf = np.stack([one[f % 3] for f in range(140)])
    monkeypatch.setenv("PA_ITEM_FRAMES", "2")
    out, info, _ = run_gpu(wl, rf, 3, rf_dtype="bf16")
    assert info["device_error_flags"] == 0
    monkeypatch.setenv("PA_ITEM_FRAMES", "1")
    ref, _, _ = run_gpu(wl, rf[:3], 3, rf_dtype="bf16")
    for f in range(140):
        assert np.array_equal(out[f], ref[f % 3]), f
