"""Batched plans hand their tasks out in an order chosen by a model of the kernel, with up to
four rings of tile buffers that consecutive frames take in turn.  Only the order differs from
frame_major plans, so every frame's result is the same, also where more frames than rings go
through (a ring's tiles are then reused) and for one, two or more groups."""
import numpy as np
import pytest

import synth
from tests.gpu_util import run_plan

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mf():
    import __graft_entry__ as g
    g.build()
    import paper_2107_06960_gb300 as mf
    return mf


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("cut,grids,size,batch", [
    (None, [(2, 3)], 64, 9),                        # one group, frames in lockstep, rings reused
    (8, [(2, 2), (1, 2)], 96, 6),
    (4, [(3, 3), (2, 2)], 32, 5),                   # tiles of one or two pixels
    ([2, 4, 8], [(2, 2), (3, 2), (2, 2), (1, 2)], 64, 5),
])
def test_batched_order_matches_frame_major(mf, dtype, cut, grids, size, batch):
    layers = synth.YOLO16
    dt = mf.BF16 if dtype == "bf16" else mf.FP32
    params = synth.make_params(layers, 3, 811, dtype)
    x = synth.make_input(batch, size, size, 3, 812, dtype)
    c, out = run_plan(mf, layers, params, x, cut, grids, dt, repeat=2)
    cm, om = run_plan(mf, layers, params, x, cut, grids, dt, plan_kwargs={"frame_major": True})
    assert np.isfinite(out).all() and np.array_equal(out, om)
    assert cut is None or np.array_equal(c, cm)
