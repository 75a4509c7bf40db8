"""Which form a launch runs, on either side of the lines.

Small launches on TMA-staged records, of records read by vector loads with few
steps, and two-frame launches with few pairs of items per SM, were measured
slower than the one-frame form; the launches next to them across each line are
not."""

import pytest

import synth

pytestmark = pytest.mark.gpu

ONE, TWO, FINE1, FINE2 = 1, 2, 3, 4


def _form(k, frames, n_elem, m, nz, dtype="f32", comp=0, ns=1024, f_number=0.0, table="lattice"):
    import torch

    import paper_2203_14906_gb300 as pa

    wl = synth.workload("cfg1", n_elem=n_elem, n_samples=ns, nx=n_elem * m, nz=nz, z1_m=nz * 0.03e-3,
                        f_number=f_number, delay_table=table, compensated=comp)
    half = n_elem * wl["pitch_m"] / 2
    wl["x0_m"], wl["x1_m"] = -half, half
    assert torch.cuda.get_device_properties(0).multi_processor_count == 152
    with pa.Plan(pa.make_desc(wl, order_k=k, rf_dtype=dtype, max_batch=frames)) as plan:
        assert plan.info()["threads"] == 128
        items = plan.info()["n_tiles"] * plan.info()["tile_x"] // 16 * frames
        return plan.form(frames), items / 152


@pytest.mark.parametrize("want,lo,hi,kw", [
    (ONE, 0, 1, dict(k=3, frames=1, n_elem=64, m=2, nz=128, dtype="bf16")),  # TMA
    (ONE, 0, 1, dict(k=3, frames=1, n_elem=64, m=2, nz=128, dtype="bf16", comp=1)),
    (ONE, 1, 2, dict(k=3, frames=3, n_elem=64, m=4, nz=128, dtype="bf16", comp=1)),
    (FINE1, 0, .5, dict(k=3, frames=1, n_elem=64, m=2, nz=128)),  # vector loads
    (FINE1, 0, .5, dict(k=3, frames=1, n_elem=40, m=2, nz=128)),
    (ONE, 0, .5, dict(k=3, frames=1, n_elem=20, m=2, nz=128)),
    (FINE1, 0, .5, dict(k=2, frames=1, n_elem=64, m=2, nz=128)),
    (ONE, 0, .5, dict(k=2, frames=1, n_elem=40, m=2, nz=128)),
    (ONE, .5, 1, dict(k=2, frames=3, n_elem=64, m=2, nz=128)),
    (FINE1, 0, .5, dict(k=6, frames=1, n_elem=64, m=2, nz=128)),
    (ONE, .5, 1, dict(k=4, frames=2, n_elem=44, m=4, nz=128)),
    (FINE1, .5, 1, dict(k=4, frames=3, n_elem=64, m=2, nz=128)),
    (FINE1, 1.5, 2, dict(k=4, frames=2, n_elem=64, m=4, nz=256, comp=1)),
    (ONE, 2, 4, dict(k=3, frames=4, n_elem=64, m=4, nz=256, comp=1)),
    (FINE1, 0, 1, dict(k=3, frames=1, n_elem=64, m=4, nz=250, ns=1022)),  # by samples
    (FINE1, 1.5, 2, dict(k=3, frames=2, n_elem=64, m=4, nz=256, ns=1022)),
    (FINE1, .5, 1, dict(k=3, frames=2, n_elem=40, m=4, nz=128, ns=1022)),
    (ONE, 1, 2, dict(k=3, frames=4, n_elem=40, m=4, nz=128, ns=1022)),
    (FINE2, 2, 4, dict(k=3, frames=4, n_elem=64, m=4, nz=256, ns=1022)),
    (ONE, 2, 4, dict(k=3, frames=4, n_elem=64, m=4, nz=256, ns=1022, comp=1)),
    (TWO, 5, 8, dict(k=3, frames=8, n_elem=64, m=4, nz=256, ns=1022)),
    (FINE1, 1, 2, dict(k=3, frames=2, n_elem=64, m=4, nz=256, table="full")),
    (FINE1, 0, 1, dict(k=7, frames=1, n_elem=64, m=4, nz=256, table="full", comp=1)),
    (ONE, 1, 2, dict(k=7, frames=2, n_elem=64, m=4, nz=256, table="full", comp=1)),
    (ONE, 0, 1, dict(k=8, frames=1, n_elem=64, m=4, nz=256, table="full", comp=1)),
    (FINE2, 2, 4, dict(k=3, frames=4, n_elem=64, m=4, nz=256, table="full")),
    (TWO, 3, 4, dict(k=2, frames=4, n_elem=64, m=4, nz=256, table="full", comp=1)),
    (ONE, 3, 4, dict(k=3, frames=4, n_elem=64, m=4, nz=256, table="full", comp=1)),
    (ONE, 6, 7.9, dict(k=2, frames=8, n_elem=64, m=4, nz=256)),  # under four pairs an SM
    (TWO, 8, 16, dict(k=2, frames=12, n_elem=64, m=4, nz=256)),
    (TWO, 6, 7.9, dict(k=3, frames=8, n_elem=64, m=4, nz=256)),
    (ONE, 3, 5.9, dict(k=3, frames=6, n_elem=64, m=4, nz=256)),
])
def test_lines(want, lo, hi, kw):
    form, per_sm = _form(**kw)
    assert lo <= per_sm <= hi, per_sm
    assert form == want, per_sm
