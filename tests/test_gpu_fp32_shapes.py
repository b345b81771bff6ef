"""The fp32 kernel's item shapes at their edges, against the fp64 oracle.

A stage's items are 16 groups of 8 pixels x 64, 32 or 16 output channels, or 8 groups x 16;
the planner picks the shape (force_nblk caps the channels).  Regions are cut into groups row
by row (row pair by row pair under a pool) or, with rect_blocks, in stacked blocks.  Every
shape sums the same products in the same order, so all of them give the same bits.

Bound per element: a chain of n = k * k * cin fused multiply-adds errs by at most
n * 2^-24 * sum |w x| (to first order, with a factor of 2 to spare for the higher orders and the
zero-padded terms), then scale, bias and leaky add a few roundings of the result.
"""
import numpy as np
import pytest

import oracle
import synth
from tests.gpu_util import run_plan

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mf():
    import __graft_entry__ as g
    g.build()
    import paper_2107_06960_gb300 as mf
    return mf


@pytest.mark.parametrize("cin,cout,k,pool,h,w,grid", [
    (3, 8, 3, False, 1, 1, (1, 1)),        # one pixel; cout below every channel block; 12-byte pixels
    (3, 32, 3, True, 34, 46, (2, 3)),      # RGB with a pool, ragged groups
    (4, 24, 3, False, 17, 9, (1, 1)),      # one quad read as 16 bytes; cout not a multiple of 16
    (16, 16, 1, False, 9, 23, (2, 1)),     # 1x1 of one chunk
    (7, 16, 3, True, 16, 18, (1, 2)),
    (8, 16, 3, True, 20, 18, (2, 2)),      # NHWC pixels of two quads
    (16, 80, 3, False, 15, 17, (1, 1)),    # cout not a multiple of 32 or 64; region 1 past a group
    (32, 64, 3, True, 8, 16, (1, 1)),      # exactly one item of 16 groups
    (48, 72, 1, False, 19, 31, (2, 2)),    # three 1x1 chunks, a channel block of 8
    (16, 128, 3, False, 130, 264, (1, 1)), # enough items for the widest shape
    (64, 64, 1, True, 146, 150, (2, 3)),
])
def test_fp32_item_shapes(mf, cin, cout, k, pool, h, w, grid):
    layers = [("conv", k, 1, (k - 1) // 2, cout)] + ([("max", 2, 2, 0, 0)] if pool else [])
    params = synth.make_params(layers, cin, 7000 + cin + cout + k, "fp32")
    x = synth.make_input(1, h, w, cin, 7100 + cin, "fp32") - np.float32(0.5)
    ref = oracle.group_outputs(layers, params, x[0], None)[-1]
    wt, sc, bi = params[0]
    mag = oracle.forward(layers[:1], [(np.abs(wt), np.ones_like(sc), np.zeros_like(bi))], np.abs(x[0]))[0]
    bound = 2.0 * (k * k * cin + 4) * 2.0 ** -24 * (np.abs(sc) * mag + np.abs(bi))
    if pool:
        hh, ww, c = bound.shape
        bound = bound.reshape(hh // 2, 2, ww // 2, 2, c).max(axis=(1, 3))
    base = None
    for kw in ({}, {"force_nblk": 64}, {"force_nblk": 32}, {"force_nblk": 16}, {"rect_blocks": True},
               {"max_ctas": 1}):
        _, out = run_plan(mf, layers, params, x, None, [grid], mf.FP32, plan_kwargs=kw)
        assert (np.abs(out[0] - ref) <= bound).all(), (kw, float((np.abs(out[0] - ref) - bound).max()))
        base = out if base is None else base
        assert np.array_equal(out, base), kw
