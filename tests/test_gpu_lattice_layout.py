"""The lattice table's order at every residue count and ragged edge.

Entries of a block of four channel steps lie together per (residue, group of
four lattice sequence numbers, depth); the cases cover residue counts with and
without common factors with the block, images ragged against the tile in both
directions, off-centre lateral ranges (lattice offsets of both signs) and
apertures of every remainder against the block, with and without apodisation.
Bar: 1e-4 of the image peak against the FP64 oracle, as for every FP32 image.
"""

import numpy as np
import pytest

import synth
from gpu_util import assert_parity, compare, oracle_frames, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n_elem,nx,nz", [(1, 29, 33, 41), (2, 30, 61, 64), (3, 31, 50, 39),
                                            (5, 24, 97, 33), (6, 17, 70, 72), (7, 19, 64, 31),
                                            (11, 22, 90, 40), (32, 16, 130, 35)])
@pytest.mark.parametrize("f_number", [0.0, 1.2])
def test_every_residue_count(m, n_elem, nx, nz, f_number):
    wl = synth.workload("cfg1", n_elem=n_elem, n_samples=512, nx=nx, nz=nz, z1_m=9e-3,
                        f_number=f_number)
    dx = wl["pitch_m"] / m
    wl["x0_m"] = -n_elem * wl["pitch_m"] / 2 + 1.3e-3
    wl["x1_m"] = wl["x0_m"] + nx * dx
    rf = synth.make_frame(wl, 3 + m)
    for k, dtype, comp in ((3, "f32", 0), (2, "bf16", 1)):
        out, info, deq = run_gpu(wl, rf, k, rf_dtype=dtype, compensated=comp)
        assert info["lattice_m"] == m and info["device_error_flags"] == 0
        assert np.isfinite(out).all()
        assert_parity(compare(out, oracle_frames(wl, deq, k)), 1e-4, what=f"m={m} k={k}")
