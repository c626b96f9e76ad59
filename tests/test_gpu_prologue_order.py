"""Softmax-GLA prologues follow one another without a barrier of the block between them: every CTA's passes give the same bits on every run, from
one chunk to several, in the forward pass, the state sweep of a recomputing backward, and the summaries of cut sequences."""
import pytest
import torch

from paper_2602_01744_b200 import api
from paper_2602_01744_b200.inputs import CONFIGS, make_inputs, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,H,d,cu", [(8, 64, 32, 128, None), (8, 130, 32, 128, None), (8, 448, 16, 64, None), (1, 2700, 16, 128, [0, 2600, 2700])])
def test_every_run_gives_the_same_bits(B, T, H, d, cu):
    cfg = small(CONFIGS["C2"], B=B, T=T, H=H, d_k=d, d_v=d, seed=3200 + T)
    x = gu.to_dev(make_inputs(cfg, with_dO=True))
    args = (x["q"], x["k"], x["v"], x["log_decay"], x["gq_logits"], x["gk_logits"])
    plan = api.sla_plan_create(cfg.variant, cfg.dtype, B, T, H, d, d)
    if cu:
        plan.set_sequences(cu)
    ws = plan.workspace(backward=True)
    runs = []
    for _ in range(12):
        o, _ = api.sla_forward(plan, *args, workspace=ws)
        g = api.sla_backward(plan, *args, x["dO"], workspace=ws)
        runs.append([o, *(t for t in g.values() if t is not None)])
    torch.cuda.synchronize()
    plan.poll()
    for other in runs[1:]:
        assert all(torch.equal(a, b) for a, b in zip(runs[0], other))
