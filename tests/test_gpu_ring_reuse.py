"""More frames than rings of tile buffers, with the tile slots of a bf16 plan sized per tile: chained
3x3 -> 1x1 pairs and explicit tile bounds give every frame the result of the frame_major plan."""
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


BOUNDS = [([0, 1, 7, 12], [0, 5, 6, 12]), ([0, 4, 6], [0, 6])]  # 12x12 cut tensor, 6x6 output


@pytest.mark.parametrize("dtype,grids,kw", [
    ("bf16", [(2, 2), (2, 1)], {"chain": True}),
    ("bf16", [(3, 3), (2, 1)], {"tile_bounds": BOUNDS}),
    ("bf16", [(3, 3), (2, 1)], {"tile_bounds": BOUNDS, "chain": True}),
    ("fp32", [(3, 3), (2, 1)], {"tile_bounds": BOUNDS}),
])
def test_reused_rings_match_frame_major(mf, dtype, grids, kw):
    layers = synth.YOLO16
    dt = mf.BF16 if dtype == "bf16" else mf.FP32
    params = synth.make_params(layers, 3, 831, dtype)
    x = synth.make_input(9, 96, 96, 3, 832, dtype)
    c, out = run_plan(mf, layers, params, x, 8, grids, dt, plan_kwargs=kw, repeat=2)
    cm, om = run_plan(mf, layers, params, x, 8, grids, dt, plan_kwargs=dict(kw, frame_major=True))
    assert np.isfinite(out).all() and np.array_equal(out, om) and np.array_equal(c, cm)
