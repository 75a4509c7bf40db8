"""The hand-over of chunks between the warps of a block.

In the two-frame and fine-grained forms the last warp out of a chunk loads the
chunk after next, from a work item that another warp may have moved on.  Short
chunks and items of one chunk make hand-overs frequent; every repetition has
the bits of the one-frame form, which stages behind block barriers.
"""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["2", "3"])
@pytest.mark.parametrize("n_elem,chunk,comp", [(8, None, 0), (61, "4", 0), (61, "4", 1), (40, "12", 0)])
def test_every_repetition_has_the_one_frame_bits(form, n_elem, chunk, comp, monkeypatch):
    import torch

    import paper_2203_14906_gb300 as pa

    frames = 24 if form == "2" else 3
    wl = synth.workload("cfg1", n_elem=n_elem, n_samples=400, nx=4 * n_elem, nz=90, z1_m=11e-3,
                        compensated=comp)
    half = n_elem * wl["pitch_m"] / 2
    wl["x0_m"], wl["x1_m"] = -half, half  # four columns a pitch, blocks of four or eight warps
    one = [synth.make_frame(wl, 20 + f) for f in range(3)]
    rf = torch.from_numpy(np.stack([one[f % 3] for f in range(frames)]).astype(np.float32)).cuda()
    if chunk:
        monkeypatch.setenv("PA_CHUNK_STEPS", chunk)
    images = {}
    for which in ("1", form):
        monkeypatch.setenv("PA_ITEM_FRAMES", which)
        with pa.Plan(pa.make_desc(wl, order_k=2, outputs=7, max_batch=frames)) as plan:
            outs = [pa.beamform(plan, rf, pa.PA_STAGE_RAW) for _ in range(1 if which == "1" else 20)]
            torch.cuda.synchronize()
            assert plan.info()["device_error_flags"] == 0
        images[which] = outs
    ref = images["1"][0]
    assert float(ref.abs().max()) > 0
    for out in images[form]:
        assert torch.equal(out, ref)
