"""How many rings of tile buffers a batched bf16 plan holds: up to four, but where the rings and the
frames' own data are more than the L2 keeps, none that the hand-out order has no use for."""
import pytest

import synth


@pytest.fixture(scope="module")
def mf():
    import __graft_entry__ as g
    g.build()
    import paper_2107_06960_gb300 as mf
    return mf


@pytest.mark.parametrize("size,cut,grids,batch,rings", [
    (608, 8, [(5, 5), (2, 2)], 4, 4),      # four frames in lockstep need their four rings
    (608, 8, [(5, 5), (2, 2)], 16, 3),     # no tile ever waits for the fourth
    (608, 8, [(5, 5), (2, 2)], 64, 3),
    (416, 8, [(3, 3), (2, 2)], 8, 4),      # small enough beside the frames
    (416, 8, [(3, 3), (2, 2)], 32, 3),
    (1216, 8, [(8, 8), (4, 4)], 8, 1),
])
def test_rings_that_crowd_the_l2_need_a_reason(mf, size, cut, grids, batch, rings):
    net = mf.Net(synth.YOLO16, size, size, 3)
    net.set_params(synth.make_params(synth.YOLO16, 3, 5, "bf16"))
    st = mf.Plan(net, cut, grids, batch=batch, dry_run=True).stats()
    ring = 0  # a slot's two buffers hold the tile's largest layer output (rounded to 128 elements)
    for g, (first, last) in enumerate([(0, cut - 1), (cut, len(synth.YOLO16) - 1)]):
        n, m = grids[g]
        ends = [l for l in range(first, last) if synth.YOLO16[l + 1][0] != "max"]  # stage ends but the group's last
        for i in range(n):
            for j in range(m):
                rects = [net.tile_region(first, last, n, m, i, j, l)[0] for l in ends]
                px = max((r[1] - r[0]) * (r[3] - r[2]) * net.shape(l)[5] for r, l in zip(rects, ends))
                ring += 2 * ((px + 127) // 128 * 128) * 2
    assert st["scratch_bytes"] == rings * ring
