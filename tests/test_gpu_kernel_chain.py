"""A call's kernels start before their predecessors end; results may not depend on it.

Calls follow one another without waiting, each on other frames and its own
images, through the graph (programmatic edges) and kernel by kernel (plain
launches); every image has the bits of the plain launches.  The cases take each
kernel of the chain: clearing or preparation pass, one-frame, two-frame and
fine-grained form, in-place, in-register and fallback post filter, log.
"""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form,k,comp,nz,frames", [
    ("1", 3, 0, 40, 1), ("1", 3, 1, 200, 3), ("1", 7, 0, 70, 2), ("2", 2, 1, 70, 3),
    ("2", 4, 0, 300, 9), ("3", 3, 0, 70, 1), ("3", 5, 1, 1100, 2)])
def test_graph_calls_in_a_row_equal_plain_launches(form, k, comp, nz, frames, monkeypatch):
    import torch

    import paper_2203_14906_gb300 as pa

    monkeypatch.setenv("PA_ITEM_FRAMES", form)
    wl = synth.workload("cfg1", n_elem=40, n_samples=700, nx=80, nz=nz, z1_m=14e-3,
                        compensated=comp)
    if not comp:  # the element lattice; otherwise the full table
        wl["x0_m"], wl["x1_m"] = -6e-3, 6e-3
    calls = 6
    rf = torch.from_numpy(np.stack(
        [[synth.make_frame(wl, 10 * c + f) for f in range(frames)] for c in range(calls)]
    ).astype(np.float32)).cuda()
    stages = pa.PA_STAGE_ENV | pa.PA_STAGE_LOG
    images = {}
    with pa.Plan(pa.make_desc(wl, order_k=k, outputs=7, max_batch=frames)) as plan:
        for graph in (True, False):
            plan.use_graph(graph)
            outs = [torch.zeros(plan.out_shape(frames, stages), device="cuda")
                    for _ in range(calls)]
            for _ in range(3):
                for c in range(calls):
                    pa.beamform(plan, rf[c], stages, out=outs[c])
            torch.cuda.synchronize()
            images[graph] = [o.cpu().numpy() for o in outs]
        assert plan.info()["device_error_flags"] == 0
    for a, b in zip(images[True], images[False]):
        assert np.array_equal(a, b) and np.abs(a).max() > 0
