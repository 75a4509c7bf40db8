"""Device memory that a plan's descriptor stands for (host logic, no GPU)."""

import paper_2203_14906_gb300 as pa
import synth


def test_slots_of_a_huge_record_are_not_wanted():
    """The prepared slots are bounded by 512 MiB: a record whose slots for one work
    item alone are larger has none (4096 channels x 65536 samples: 4.3 GB)."""
    wl = synth.workload("cfg1", n_elem=4096, n_samples=65536, nx=64, nz=64, z1_m=10e-3,
                        pitch_m=1e-5, x0_m=-0.32e-3, x1_m=0.32e-3)
    for frames in (1, 2, 8):
        assert pa.footprint(pa.make_desc(wl, order_k=3, max_batch=frames), 0) < 256 << 20
