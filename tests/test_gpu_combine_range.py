"""e_k over the FP32 range: two-float arithmetic inside, FP64 outside it.

The fused kernel forms e_k in two-float arithmetic while a pixel's amplitude
sum lies in (2^-60, 2^40) and in FP64 beyond.  The same frame is scaled so that
its images fall inside, outside and across both ends of that interval; e_k is
homogeneous of degree one in the RF, so the bar (1e-4 of the image peak, as
for every FP32 image) is the same at every scale.
"""

import numpy as np
import pytest

import synth
from gpu_util import assert_parity, compare, oracle_frames, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("exponent", [-75, -66, -63, 0, 33, 36, 60])
def test_raw_images_at_every_scale(k, exponent):
    wl = synth.workload("cfg1", n_elem=32, n_samples=768, nx=64, nz=64, z1_m=12e-3)
    wl["x0_m"], wl["x1_m"] = -32 * 0.15e-3, 32 * 0.15e-3
    rf = synth.make_frame(wl, 6)
    rf = rf / np.sqrt(np.mean(rf * rf)) * 2.0 ** exponent
    out, info, deq = run_gpu(wl, rf, k, stages=1)
    assert info["device_error_flags"] == 0 and np.isfinite(out).all()
    refs = oracle_frames(wl, deq, k, stages=("raw",))
    assert_parity(compare(out, refs, stages=1), 1e-4, what=f"k={k} 2^{exponent}")
    # the amplitude sums of the scaled frames: 2^exponent times about 32
    if exponent in (-63, 36):
        sums = np.abs(deq).mean() * 32
        edge = 2.0 ** (-60 if exponent < 0 else 40)
        assert edge / 64 < sums < edge * 64


def test_silent_frame_gives_zeros():
    wl = synth.workload("cfg1", n_elem=32, n_samples=768, nx=64, nz=64, z1_m=12e-3)
    for k in (3, 4, 5, 8):
        out, _, _ = run_gpu(wl, np.zeros((32, 768)), k, stages=1)
        assert not out.any()
