"""e_k of very large apertures whose terms leave FP32's range.

With N channels of one amplitude a, e_8 = C(N, 8) a, and the terms of Newton's
identities are larger by up to 8! / 7!..: at 24 000 channels of 2^25 the result is
finite in FP32 and a term is not.  Such pixels take the FP64 form; below the line
the two-float form agrees as well.  Kahan sums keep the sums' own error far under
the bar of 1e-4.
"""

from math import comb

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [25.3, 10.0])
def test_order_8_of_24000_channels(exponent):
    import torch

    import paper_2203_14906_gb300 as pa

    n, a = 24000, np.float32(2.0 ** exponent)
    wl = synth.workload("cfg1", n_elem=n, n_samples=1024, nx=32, nz=32, pitch_m=2e-6, x0_m=-32e-6,
                        x1_m=32e-6, z0_m=2e-3, z1_m=4e-3, compensated=1)
    want = float(comb(n, 8)) * float(a)
    assert want < 3.4e38 and n * a < 2.0 ** 40
    rf = torch.full((1, n, 1024), float(a), dtype=torch.float32, device="cuda")
    with pa.Plan(pa.make_desc(wl, order_k=8, outputs=pa.PA_OUT_HODMAS)) as plan:
        out = pa.beamform(plan, rf, pa.PA_STAGE_RAW).double()
        assert plan.info()["device_error_flags"] == 0
    err = float((out / want - 1.0).abs().max())
    assert err <= 1e-4, err
