"""Batched fp32 plans may hold up to four rings of tile buffers.  More rings never take a plan
over the 32 MiB of the allocation-free entry point: where the plan fits with one ring
(frame_major), it fits with the rings that the planner chose."""
import pytest

import synth

AREA = 32 << 20


@pytest.fixture(scope="module")
def mf():
    import __graft_entry__ as g
    g.build()
    import paper_2107_06960_gb300 as mf
    return mf


def _r256(x):
    return (x + 255) // 256 * 256


def _need(mf, cuts, grids, batch, **kw):
    layers = synth.YOLO16
    net = mf.Net(layers, 96, 96, 3)
    net.set_params(synth.make_params(layers, 3, 5, "fp32"))
    st = mf.Plan(net, cuts, grids, batch=batch, dtype=mf.FP32, dry_run=True, **kw).stats()
    sh = net.shape((cuts[0] if isinstance(cuts, list) else cuts) - 1)
    counters = 4 + st["n_tasks"] + batch * len(grids)
    return _r256(4 * counters) + _r256(4 * batch * sh[3] * sh[4] * sh[5]) + _r256(st["scratch_bytes"]), st


@pytest.mark.parametrize("cuts,grids,batches", [
    (2, [(1, 1), (1, 1)], (8, 90, 96, 100, 104)),          # the cut tensor takes most of the area
    (8, [(2, 2), (2, 2)], (2, 64, 300, 360)),
    ([2, 4, 8], [(1, 1), (1, 1), (1, 1), (2, 2)], (4, 48, 56, 62, 64)),
])
def test_rings_leave_fitting_plans_in_the_area(mf, cuts, grids, batches):
    fits = 0
    for b in batches:
        one, _ = _need(mf, cuts, grids, b, frame_major=True)
        many, _ = _need(mf, cuts, grids, b)
        assert many >= one
        if one <= AREA:
            fits += 1
            assert many <= AREA, (b, one, many)
        else:
            assert many == one
    assert fits >= 2
