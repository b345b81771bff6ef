"""weight_bytes of an fp32 plan is what it holds: weights packed in chunks of input channels (4 of a
3x3 convolution, 16 of a 1x1) and whole blocks of output channels (16 here), with scale and bias."""
import numpy as np
import pytest


@pytest.fixture(scope="module")
def mf():
    import __graft_entry__ as g
    g.build()
    import paper_2107_06960_gb300 as mf
    return mf


@pytest.mark.parametrize("k,cin,cout,pad_in,pad_out", [
    (3, 3, 8, 4, 16),
    (3, 6, 24, 8, 32),
    (1, 48, 40, 48, 48),
    (3, 32, 64, 32, 64),     # nothing to pad
])
def test_weight_bytes_counts_the_padding(mf, k, cin, cout, pad_in, pad_out):
    net = mf.Net([("conv", k, 1, k // 2, cout)], 12, 12, cin)
    net.set_weights(0, np.zeros((cout, cin, k, k)), np.ones(cout), np.zeros(cout))
    st = mf.Plan(net, None, [(1, 1)], dtype=mf.FP32, dry_run=True, force_nblk=16).stats()  # blocks of 16 channels
    assert st["weight_bytes"] == 4 * pad_in * k * k * pad_out + 2 * 4 * pad_out
