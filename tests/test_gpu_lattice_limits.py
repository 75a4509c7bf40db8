"""The largest lattice tables: one row per lattice offset, near 2^16 rows.

A table of 65 534 rows (32 columns and 65 497 elements on one column a pitch, with
the padding rows of either layout between 65 534 and 65 540) builds, and DAS of a
constant record is the channel count times the constant."""

import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [65481, 65497, 70001])
def test_tables_of_65_thousand_rows(n):
    import torch

    import paper_2203_14906_gb300 as pa

    wl = synth.workload("cfg1", n_elem=n, n_samples=256, nx=32, nz=40, pitch_m=1e-7, x0_m=-1.6e-6,
                        x1_m=1.6e-6, z0_m=2e-3, z1_m=5e-3, compensated=1)
    rf = torch.full((1, n, 256), 0.5, dtype=torch.float32, device="cuda")
    with pa.Plan(pa.make_desc(wl, order_k=2, outputs=pa.PA_OUT_DAS)) as plan:
        assert plan.info()["lattice_m"] == 1
        out = pa.beamform(plan, rf, pa.PA_STAGE_RAW)
        assert plan.info()["device_error_flags"] == 0
    assert float((out / (0.5 * n) - 1.0).abs().max()) <= 1e-6
