"""A server's device budget, fixed in bytes.

A plan of this workload cannot do without 4.5 MB (its tables); its prepared slots,
18 MB at eight frames a batch, are extra and may not cost a request its admission
or another plan its place."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

RAW = 1
MB = 1 << 20


def _frames(wl, n):
    import torch

    return [torch.from_numpy(synth.make_frame(wl, 40 + s).astype(np.float32)).pin_memory() for s in range(n)]


def _serve(wl, orders, frames, budget, **kw):
    """Batches of all frames of each order in turn, twice over, one order at a time."""
    import torch

    import paper_2203_14906_gb300 as pa
    from paper_2203_14906_gb300.serving import Server

    outs = {}
    with Server(budget_bytes=budget, stages=RAW, **kw) as srv:
        for rep in range(2):
            for k in orders:
                desc = pa.make_desc(wl, order_k=k, outputs=1)
                outs[k] = [torch.zeros((1, 1, wl["nx"], wl["nz"])).pin_memory() for _ in frames]
                ts = [srv.submit(desc, f.data_ptr(), o.data_ptr()) for f, o in zip(frames, outs[k])]
                assert all(srv.wait(t, timeout_ms=60000)["status"] == 0 for t in ts)
                assert srv.stats()["bytes_peak"] <= budget
        st = srv.stats()
    for k in orders:
        with pa.Plan(pa.make_desc(wl, order_k=k, outputs=1)) as plan:
            for f, o in zip(frames, outs[k]):
                want = pa.beamform(plan, f.cuda()[None], RAW).cpu()[0]
                assert torch.equal(o, want), k
    return st


@pytest.mark.parametrize("budget_mb", [35, 64])  # no room for slots; room for two plans' slots
def test_slots_cost_no_plan_its_place(budget_mb):
    """Four plans and one batch of eight frames (16 MB) fit without slots."""
    wl = synth.workload("cfg2")
    st = _serve(wl, (3, 2, 4, 5), _frames(wl, 8), budget_mb * MB, slots=1, max_batch=8)
    assert st["plans_resident"] == 4


def test_slots_are_taken_where_the_budget_has_them():
    wl = synth.workload("cfg2")
    frames = _frames(wl, 8)
    st = _serve(wl, (3,), frames, 64 * MB, slots=1, max_batch=8)
    assert st["bytes_in_use"] > 20 * MB


@pytest.mark.parametrize("budget_mb,slots", [(12, 1), (12, 2), (20, 2), (40, 3)])
def test_a_batch_larger_than_the_budget_is_cut(budget_mb, slots):
    """A plan and eight frames' buffers (4.5 + 16 MB) do not fit in the two smaller
    budgets: the batch is cut, and the plan about to run is not evicted for its own
    buffers.  The larger ones evict one plan for another."""
    wl = synth.workload("cfg2")
    _serve(wl, (3, 2, 4), _frames(wl, 8), budget_mb * MB, slots=slots, max_batch=8)


def test_mixed_orders_under_a_tight_budget():
    """Requests of several plans at once, two batches in flight, room for two plans."""
    import torch

    import paper_2203_14906_gb300 as pa
    from paper_2203_14906_gb300.serving import Server

    wl = synth.workload("cfg2")
    frames = _frames(wl, 4)
    with Server(budget_bytes=24 * MB, stages=RAW, slots=2, max_batch=4) as srv:
        jobs = []
        for i in range(24):
            k, f = 2 + i % 3, frames[i % 4]
            o = torch.zeros((1, 1, wl["nx"], wl["nz"])).pin_memory()
            jobs.append((k, f, o, srv.submit(pa.make_desc(wl, order_k=k, outputs=1), f.data_ptr(), o.data_ptr())))
        assert all(srv.wait(j[3], timeout_ms=60000)["status"] == 0 for j in jobs)
        assert srv.stats()["bytes_peak"] <= 24 * MB
    for k in (2, 3, 4):
        with pa.Plan(pa.make_desc(wl, order_k=k, outputs=1)) as plan:
            want = [pa.beamform(plan, f.cuda()[None], RAW).cpu()[0] for f in frames]
        assert all(torch.equal(o, want[i % 4]) for i, (kk, f, o, t) in enumerate(jobs) if kk == k)
