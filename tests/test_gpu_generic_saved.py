"""fp32 kernels and SLA_FLAG_SAVE_FOR_BACKWARD: a backward on the workspace a forward was given skips its recomputation, with the same bits;
other inputs, another workspace, or a forward on scratch of its own size recompute."""
import pytest
import torch

from paper_2602_01744_b200 import api
from paper_2602_01744_b200.inputs import CONFIGS, make_inputs, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base,T,dk,dv", [("C0", 130, 64, 64), ("C1", 65, 48, 96), ("C4", 200, 64, 32)])
def test_backward_reads_what_the_forward_left_only_where_it_was_kept(base, T, dk, dv):
    cfg = small(CONFIGS[base], B=2, T=T, H=3, d_k=dk, d_v=dv, dtype="fp32", seed=2200 + T, backward=True)
    x = gu.to_dev(make_inputs(cfg, with_dO=True, with_h0=True))
    args = (x["q"], x["k"], x["v"], x["log_decay"], x["gq_logits"], x["gk_logits"])
    plan = api.sla_plan_create(cfg.variant, cfg.dtype, cfg.B, cfg.T, cfg.H, dk, dv, flags=api.SLA_FLAG_SAVE_FOR_BACKWARD)
    plain = api.sla_plan_create(cfg.variant, cfg.dtype, cfg.B, cfg.T, cfg.H, dk, dv)
    assert plan.forward_workspace_bytes == plain.forward_workspace_bytes < plan.backward_workspace_bytes
    ws, ws2 = plan.workspace(backward=True), plan.workspace(backward=True)

    def backward(p, w, k=x["k"]):
        g = api.sla_backward(p, x["q"], k, *args[2:], x["dO"], beta=x["beta"], h0=x["h0"], dht=x["dht"], want_dh0=True, workspace=w)
        return g, p.last_launch_count

    forward = lambda w: api.sla_forward(plan, *args, beta=x["beta"], h0=x["h0"], workspace=w)
    ref, full = backward(plain, ws2)
    forward(ws)
    got = [backward(plan, ws), backward(plan, ws)]                # read what was left, both times
    assert got[0][1] == got[1][1] < full
    got += [backward(plan, ws2), backward(plan, ws, x["k"].clone()), backward(plan, ws)]     # another workspace; other inputs, which overwrite
    forward(ws[:plan.forward_workspace_bytes])
    got.append(backward(plan, ws))                                # scratch of the forward's own size: not kept
    assert [n for _, n in got[2:]] == [full] * 4
    torch.cuda.synchronize()
    plan.poll()
    for g, _ in got:
        for n, t in ref.items():
            if t is not None:
                assert torch.equal(t, g[n]), n
