"""Packed sums of the two-frame form: every kernel variant with the element
lattice (order, apodisation, Kahan sums, samples) gives the one-frame form's bits,
on an odd frame count and with a silent frame (zero sums)."""

import itertools

import numpy as np
import pytest

import synth
from gpu_util import run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 2, 3, 4, 5])
def test_every_variant_has_the_one_frame_bits(k, monkeypatch):
    for f_number, comp, interp in itertools.product((0.0, 1.5), (0, 1), ("linear", "nearest")):
        wl = synth.workload("cfg1", n_elem=72, n_samples=400, nx=144, nz=70, z1_m=13e-3,
                            f_number=f_number, interp=interp)
        wl["x0_m"], wl["x1_m"] = -72 * 0.15e-3, 72 * 0.15e-3
        rf = np.stack([synth.make_frame(wl, 30 + f) for f in range(3)])
        rf[1] = 0.0
        outs = []
        for form in ("1", "2"):
            monkeypatch.setenv("PA_ITEM_FRAMES", form)
            out, info, _ = run_gpu(wl, rf, k, compensated=comp, stages=1)
            assert info["device_error_flags"] == 0
            outs.append(out)
        assert np.array_equal(*outs), (f_number, comp, interp)
        assert not outs[1][1].any() and np.abs(outs[1][2]).max() > 0
