"""The measured search sizes (and times) the plan that its caller gets by building a candidate:
with a batch, the default plan with its rings of tiles, or one ring where those are over the
budget, which the candidate names in ring_slots."""
import pytest

import synth


@pytest.fixture(scope="module")
def mf():
    import __graft_entry__ as g
    g.build()
    import paper_2107_06960_gb300 as mf
    return mf


def _bytes(mf, net, c, batch, dtype, **kw):
    st = mf.Plan(net, c["cut"], c["grids"], batch=batch, dtype=dtype, dry_run=True, **kw).stats()
    esz = 2 if dtype == mf.BF16 else 4
    cut = 0
    if c["cut"] is not None:
        sh = net.shape(c["cut"] - 1)
        cut = batch * ((sh[5] + 7) // 8 * 8) * sh[3] * sh[4] * esz
    return st["scratch_bytes"] + cut, st


@pytest.mark.parametrize("dtype,size,batch", [("bf16", 608, 4), ("bf16", 224, 16), ("fp32", 96, 3)])
def test_candidate_bytes_are_those_of_the_plan_it_names(mf, dtype, size, batch):
    dt = mf.BF16 if dtype == "bf16" else mf.FP32
    net = mf.Net(synth.YOLO16, size, size, 3)
    net.set_params(synth.make_params(synth.YOLO16, 3, 5, dtype))
    kw = dict(cuts=(8,), max_grid=2, dry_run=True, batch=batch, dtype=dt)
    free, _ = net.search_measured(budget_bytes=-1, **kw)
    for c in free:
        want, st = _bytes(mf, net, c, batch, dt)
        assert c["status"] == 0 and c["ring_slots"] == 0 and c["intermediate_bytes"] == want
        assert c["executed_flops"] == st["executed_flops"]
    ring = [_bytes(mf, net, c, batch, dt, ring_slots=_bytes(mf, net, c, batch, dt)[1]["ring_slots"])[0] for c in free]
    budget = sorted(ring)[len(ring) // 2]
    capped, _ = net.search_measured(budget_bytes=budget, **kw)
    for c, one, f in zip(capped, ring, free):
        assert c["intermediate_bytes"] == _bytes(mf, net, c, batch, dt, ring_slots=c["ring_slots"])[0]
        # no candidate that fits, with its default rings or with one, is refused
        assert c["status"] == (0 if min(f["intermediate_bytes"], one) <= budget else mf.ENOFIT)
        assert (c["ring_slots"] > 0) == (one <= budget < f["intermediate_bytes"])
    assert any(c["ring_slots"] > 0 for c in capped) and any(c["status"] == mf.ENOFIT for c in capped)
