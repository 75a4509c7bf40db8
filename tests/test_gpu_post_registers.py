"""The register-resident post-filter kernel at its edges.

Launches of many column pairs of 256-1024 points keep the transforms in
registers.  Depths just above and at powers of two (most and no zero padding),
odd column counts (a pair with one column), and every kind of band: the default
ones, one of a few bins, a wide one, the analytic mask alone (all positive bins,
DC and M/2) and a band above the axial Nyquist rate (DC removal).  Envelopes are
held to the oracle (1e-4 of the peak, LOG 0.05 dB near it), and a silent image
gives zeros and the clipping range.
"""

import numpy as np
import pytest

import synth
from gpu_util import assert_parity, compare, oracle_frames, run_gpu

pytestmark = pytest.mark.gpu

BANDS = {"default": (0.0, 0.0), "narrow": (3.0e6, 3.2e6), "wide": (0.3e6, 9.0e6), "off": (0.0, -1.0),
         "above": (60e6, 70e6)}


@pytest.mark.parametrize("nz", [129, 256, 257, 511, 512, 513, 1000])
@pytest.mark.parametrize("band", sorted(BANDS))
def test_envelopes(nz, band):
    lo, hi = BANDS[band]
    wl = synth.workload("cfg1", n_elem=16, n_samples=640, nx=161, nz=nz, z1_m=nz * 0.02e-3,
                        band_lo_hz=lo, band_hi_hz=hi)
    wl["x0_m"], wl["x1_m"] = -16 * 0.15e-3, -16 * 0.15e-3 + 161 * 0.03e-3
    m = 256 if nz <= 256 else 512 if nz <= 512 else 1024
    frames = 32 * 1100 // (m // 32) // (81 * 3) + 1  # past the register kernel's line
    one = np.stack([synth.make_frame(wl, 5), np.zeros((16, 640))])
    rf = one[np.arange(frames) % 2]
    out, info, deq = run_gpu(wl, rf, 2, stages=6)
    assert info["fft_size"] == m and info["device_error_flags"] == 0
    if band != "above":
        refs = oracle_frames(wl, deq[:1], 2)
        assert_parity(compare(out[:1], refs, stages=6), 1e-4, what=f"{nz} {band}")
    else:
        env = oracle_frames(wl, deq[:1], 2)[0]["env"]
        for o, name in enumerate(("das", "dmas", "ho")):
            assert np.max(np.abs(out[0, 0, o] - env[name])) <= 1e-4 * np.max(env[name])
    for f in range(2, frames):
        assert np.array_equal(out[f], out[f % 2])
    assert not out[1, 0].any() and (out[1, 1] == -60.0).all()
