"""A fused max-pool takes the vertical maximum of the accumulators before it applies scale, bias,
leaky ReLU and rounding, with the sign of every channel's scale moved into its weights.  Channels
of negative, zero and mixed scales, at output channel counts of 32-column and 16-column units and
with the last octets past cout, against the oracle: rounding is monotonic, so the bound is that of
any single bf16 layer, half an ulp of the result and the accumulation's error (fp32: 2^-18 covers
576 products)."""
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


@pytest.mark.parametrize("cin,cout,k,h,w,grid,dtype", [
    (3, 32, 3, 36, 40, (2, 3), "bf16"),    # gathered first layer, blocks across columns
    (3, 8, 3, 20, 24, (1, 1), "bf16"),     # N = 16
    (32, 24, 3, 34, 30, (2, 2), "bf16"),   # N = 32, an octet past cout
    (64, 40, 3, 26, 42, (1, 2), "bf16"),   # N = 48: 16-column units
    (64, 256, 1, 32, 18, (2, 1), "bf16"),  # eight units per block
    (16, 96, 3, 130, 34, (1, 1), "bf16"),  # three units per block, several blocks an item
    (16, 40, 3, 22, 26, (1, 2), "fp32"),   # the fp32 kernel keeps the scales as they are
])
def test_pooled_scale_signs(mf, cin, cout, k, h, w, grid, dtype):
    layers = [("conv", k, 1, (k - 1) // 2, cout), ("max", 2, 2, 0, 0)]
    (wt, sc, bi), _ = synth.make_params(layers, cin, 9100 + cout, dtype)
    sc = sc.copy()
    sc[0::4] *= -1.0
    sc[1::8] = 0.0
    sc[5::8] = -0.0
    params = [(wt, sc, bi), None]
    x = synth.make_input(1, h, w, cin, 9200 + cin, dtype) - np.float32(0.5)
    if dtype == "bf16":
        x = synth.round_bf16(x)
    ref = oracle.group_outputs(layers, params, x[0], None)[-1]
    _, out = run_plan(mf, layers, params, x, None, [grid], mf.BF16 if dtype == "bf16" else mf.FP32)
    eps = 2.0 ** -8 if dtype == "bf16" else 2.0 ** -18
    bound = eps * np.abs(ref) + (2.0 ** -12 if dtype == "bf16" else 2.0 ** -18) * np.abs(ref).max()
    bad = np.abs(out[0] - ref) > bound
    assert not bad.any(), "%d of %d out of bound, worst %.3g" % (bad.sum(), bad.size, np.abs(out[0] - ref).max())
