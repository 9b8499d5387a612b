"""wino_debug_dump_stage copies what the most recent call left in its workspace, or refuses: it reads no
buffer that the caller may have reused since, and returns nothing of an earlier call."""
import numpy as np
import pytest

import oracle
import wino_inputs as wi
from helpers import build_layer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [2, 4, 6])
def test_no_stages_of_a_one_launch_call(m):
    import torch
    from paper_2002_10711_b200 import binding
    from paper_2002_10711_b200.layer import WinogradConv
    L, x_q, w_q, bias = build_layer(wi.Workload("du", 5800 + m, 2, 64, 7, 9, 80, m))
    _, want = oracle.forward(L, x_q, w_q, bias=bias, dumps=True)
    plan = binding.Plan.from_layer(L)
    conv = WinogradConv(plan)
    conv.load_weights(w_q, bias)
    x = torch.from_numpy(np.ascontiguousarray(x_q)).cuda()
    stages = ((binding.STAGE_VQ, "V_q"), (binding.STAGE_M_I32, "M"), (binding.STAGE_MQ, "m_q"))
    for first in (True, False):                # also after a call that did leave its stages
        before = plan.launch_count
        y = conv.forward(x)
        assert plan.launch_count - before == 1
        for stage, _ in stages:
            with pytest.raises(binding.WinoError) as e:
                conv.dump(stage)
            assert e.value.code == binding.ERR_UNSUPPORTED
        if first:                              # the way to see them, on the caller's own x
            y2 = conv.empty_output()
            plan.debug_run_stages(7, x, conv.Uq, conv.bias, y2, conv.ws)
            assert torch.equal(y, y2)
            for stage, name in stages:
                assert (conv.dump(stage).cpu().numpy().reshape(-1) == want[name].reshape(-1)).all()
    assert plan.last_status() == 0


def test_no_stage_of_an_earlier_call_after_a_call_without_workspace():
    import torch
    from paper_2002_10711_b200 import binding
    from paper_2002_10711_b200.layer import WinogradConv
    L, x_q, w_q, bias = build_layer(wi.Workload("du", 5810, 160, 64, 16, 16, 64, 2))
    plan = binding.Plan.from_layer(L)
    assert plan.path == binding.PATH_FUSED_F2
    conv = WinogradConv(plan)
    conv.load_weights(w_q, bias)
    x = torch.from_numpy(np.ascontiguousarray(x_q)).cuda()
    conv.forward(x)                            # with a workspace: the staged kernels
    conv.dump(binding.STAGE_VQ)
    plan.conv_forward(x, conv.Uq, conv.bias, conv.empty_output(), None)
    with pytest.raises(binding.WinoError) as e:
        conv.dump(binding.STAGE_VQ)
    assert e.value.code == binding.ERR_UNSUPPORTED
