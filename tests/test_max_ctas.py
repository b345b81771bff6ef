"""options.max_ctas above the SM count: the tensor-core kernel's first items go out by CTA index,
so a bf16 plan takes no more CTAs than can be resident (one per SM)."""
import numpy as np
import pytest

import synth


@pytest.fixture(scope="module")
def mf():
    import __graft_entry__ as g
    g.build()
    import paper_2107_06960_gb300 as mf
    return mf


def _net(mf, size):
    net = mf.Net(synth.YOLO16, size, size, 3)
    net.set_params(synth.make_params(synth.YOLO16, 3, 9, "bf16"))
    return net


@pytest.mark.parametrize("max_ctas", [153, 608, 2**30])
def test_items_are_shaped_for_resident_ctas(mf, max_ctas):
    net = _net(mf, 608)
    grids = [(5, 5), (2, 2)]
    default = mf.Plan(net, 8, grids, dry_run=True).stats()
    st = mf.Plan(net, 8, grids, dry_run=True, max_ctas=max_ctas).stats()
    assert st["n_items"] == default["n_items"] and st["issued_flops"] == default["issued_flops"]


@pytest.mark.gpu
def test_more_ctas_than_sms_run_as_one_per_sm(mf):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    net = _net(mf, 224)
    x = torch.from_numpy(synth.make_input(1, 224, 224, 3, 10, "bf16")).bfloat16().cuda()
    outs = []
    for max_ctas in (0, sms + 1, 4 * sms):
        plan = mf.Plan(net, 8, [(5, 5), (2, 2)], max_ctas=max_ctas)
        assert plan.stats()["max_ctas"] == sms
        out = torch.full((1,) + net.shape(15)[3:], float("nan"), dtype=torch.bfloat16, device="cuda")
        plan.run(x, out)
        plan.sync_status(like=x)
        outs.append(out.float().cpu().numpy())
        plan.close()
    assert np.isfinite(outs[0]).all() and np.array_equal(outs[0], outs[1]) and np.array_equal(outs[0], outs[2])
