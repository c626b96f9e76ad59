"""A sequence table that is refused leaves the plan with the one it had, and with the sizes that belong to it."""
import ctypes

import pytest
import torch

from paper_2602_01744_b200 import api
from paper_2602_01744_b200.inputs import CONFIGS, make_inputs, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


# (as one regular batch the first of them runs in segments, with scratch that the packed batch does not ask for)
@pytest.mark.parametrize("base,T,flags", [("C1", 2600, 0), ("C2", 700, api.SLA_FLAG_SAVE_FOR_BACKWARD), ("C4", 1300, 0)])
def test_a_refused_table_changes_nothing(base, T, flags):
    cfg = small(CONFIGS[base], B=1, T=T, H=2, seed=3000 + T)
    x = gu.to_dev(make_inputs(cfg))
    args = (x["q"], x["k"], x["v"], x["log_decay"], x["gq_logits"], x["gk_logits"])
    plan = api.sla_plan_create(cfg.variant, cfg.dtype, 1, T, 2, cfg.d_k, cfg.d_v, flags=flags)
    good = [*range(0, T, 130), T]

    def sizes():
        f, b = ctypes.c_size_t(), ctypes.c_size_t()
        assert api.lib().sla_plan_workspace_bytes(plan.handle, ctypes.byref(f), ctypes.byref(b)) == 0
        return f.value, b.value

    regular = sizes()
    plan.set_sequences(good)
    packed = sizes()
    o, _ = api.sla_forward(plan, *args, beta=x["beta"])
    for bad in ([0, T + 1], [1, T], [0, 7, 7, T], [0, 9, 5, T]):
        with pytest.raises(api.SLAError):
            plan.set_sequences(bad)
        assert sizes() == packed == (plan.forward_workspace_bytes, plan.backward_workspace_bytes)
        o2, _ = api.sla_forward(plan, *args, beta=x["beta"])
        assert torch.equal(o, o2)
    torch.cuda.synchronize()
    plan.poll()
    plan.set_sequences(None)
    assert sizes() == regular
    with pytest.raises(api.SLAError):                             # a plan without a table stays without one
        plan.set_sequences([0, 3])
    assert sizes() == regular
