"""A captured forward pass over a packed batch replays what it was captured with, whatever backward passes of the same plan read in between."""
import pytest
import torch

from paper_2602_01744_b200 import api
from paper_2602_01744_b200.inputs import CONFIGS, make_inputs, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base", ["C2", "R2"])
def test_a_backward_pass_on_other_tensors_between_replays(base):
    cu, H = [0, 2600, 2700], 2                                    # (the long sequence is cut, forward and backward)
    cfg = small(CONFIGS[base], B=1, T=cu[-1], H=H, seed=3100)
    xs = [gu.to_dev(make_inputs(small(cfg, seed=3100 + i), with_dO=True)) for i in range(2)]
    args = [(x["q"], x["k"], x["v"], x["log_decay"], x["gq_logits"], x["gk_logits"]) for x in xs]
    plan = api.sla_plan_create(cfg.variant, cfg.dtype, 1, cfg.T, H, cfg.d_k, cfg.d_v)
    plan.set_sequences(cu)
    ws, ws2 = plan.workspace(), plan.workspace(backward=True)
    o, ht = torch.empty_like(xs[0]["v"]), torch.empty(2, H, cfg.d_k, cfg.d_v, device="cuda")
    forward = lambda: api.sla_forward(plan, *args[0], o=o, ht=ht, workspace=ws)
    forward()
    assert plan.last_launch_count == 3
    ref = o.clone(), ht.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        forward()
    api.sla_backward(plan, *args[1], xs[1]["dO"], workspace=ws2)
    o.fill_(0)
    ht.fill_(0)
    graph.replay()
    torch.cuda.synchronize()
    plan.poll()
    assert torch.equal(o, ref[0]) and torch.equal(ht, ref[1])
    del graph
