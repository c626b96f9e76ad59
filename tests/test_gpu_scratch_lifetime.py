"""Calls from Python that bring no workspace: their scratch goes back to the allocator, other tensors take its place, and a backward pass that is
handed the same memory again must not find anything there."""
import pytest
import torch

from paper_2602_01744_b200 import api
from paper_2602_01744_b200.inputs import CONFIGS, make_inputs, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


# Softmax-GLA and -RetNet, the chunk-parallel Softmax-GatedDeltaNet kernels and their one-CTA form
@pytest.mark.parametrize("base,T", [("C2", 200), ("R2", 200), ("C4", 1100), ("C4", 200)])
def test_a_saving_forward_without_a_workspace_leaves_nothing_to_rely_on(base, T):
    cfg = small(CONFIGS[base], B=1, T=T, H=2, seed=2900 + T)
    x = gu.to_dev(make_inputs(cfg, with_dO=True))
    args = (x["q"], x["k"], x["v"], x["log_decay"], x["gq_logits"], x["gk_logits"])
    create = lambda flags: api.sla_plan_create(cfg.variant, cfg.dtype, 1, T, 2, cfg.d_k, cfg.d_v, flags=flags)
    ref = api.sla_backward(create(0), *args, x["dO"], beta=x["beta"])
    plan, out = create(api.SLA_FLAG_SAVE_FOR_BACKWARD), {n: None if t is None else torch.empty_like(t) for n, t in ref.items()}
    o = torch.empty_like(x["v"])
    api.sla_forward(plan, *args, beta=x["beta"], o=o)
    other = torch.full((plan.forward_workspace_bytes,), 255, dtype=torch.uint8, device="cuda")      # where the scratch was: NaN
    del other
    got = [api.sla_backward(plan, *args, x["dO"], beta=x["beta"], out=out)]
    ws = plan.workspace(backward=True)                            # a workspace of the caller's own is relied on as ever
    api.sla_forward(plan, *args, beta=x["beta"], workspace=ws)
    full = plan.last_launch_count
    got.append(api.sla_backward(plan, *args, x["dO"], beta=x["beta"], workspace=ws))
    assert (full, plan.last_launch_count) == (1, 2)
    torch.cuda.synchronize()
    plan.poll()
    for g in got:
        for n, t in ref.items():
            if t is not None:
                assert torch.equal(t, g[n]), n


@pytest.mark.parametrize("base,T", [("C2", 200), ("C4", 1100)])
def test_a_backward_without_a_workspace_does_not_rely_on_one_that_is_gone(base, T):
    cfg = small(CONFIGS[base], B=1, T=T, H=2, seed=2950 + T)
    x = gu.to_dev(make_inputs(cfg, with_dO=True))
    args = (x["q"], x["k"], x["v"], x["log_decay"], x["gq_logits"], x["gk_logits"])
    create = lambda flags: api.sla_plan_create(cfg.variant, cfg.dtype, 1, T, 2, cfg.d_k, cfg.d_v, flags=flags)
    ref = api.sla_backward(create(0), *args, x["dO"], beta=x["beta"])
    plan, out = create(api.SLA_FLAG_SAVE_FOR_BACKWARD), {n: None if t is None else torch.empty_like(t) for n, t in ref.items()}
    o = torch.empty_like(x["v"])
    ws = plan.workspace(backward=True)
    api.sla_forward(plan, *args, beta=x["beta"], o=o, workspace=ws)
    n = ws.numel()
    del ws
    other = torch.full((n,), 255, dtype=torch.uint8, device="cuda")
    del other
    g = api.sla_backward(plan, *args, x["dO"], beta=x["beta"], out=out)
    torch.cuda.synchronize()
    plan.poll()
    for name, t in ref.items():
        if t is not None:
            assert torch.equal(t, g[name]), name
