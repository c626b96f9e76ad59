"""fp32 kernels and SLA_FLAG_SAVE_FOR_BACKWARD, which they ignore: a backward pass recomputes whatever became of the workspace since the forward
pass - taken by another layer's plan, or written over - and gives the bits of a plan without the flag."""
import pytest
import torch

from paper_2602_01744_b200 import api
from paper_2602_01744_b200.inputs import CONFIGS, make_inputs, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base,T,dk,dv", [("C0", 130, 64, 64), ("C1", 65, 48, 96), ("C4", 200, 64, 32)])
def test_layers_that_share_one_workspace(base, T, dk, dv):
    cfg = small(CONFIGS[base], B=2, T=T, H=3, d_k=dk, d_v=dv, dtype="fp32", seed=2200 + T, backward=True)
    layers = [gu.to_dev(make_inputs(small(cfg, seed=cfg.seed + i), with_dO=True, with_h0=True)) for i in range(2)]
    create = lambda flags: api.sla_plan_create(cfg.variant, cfg.dtype, cfg.B, cfg.T, cfg.H, dk, dv, flags=flags)
    plans, plain = [create(api.SLA_FLAG_SAVE_FOR_BACKWARD) for _ in layers], create(0)
    ws = plain.workspace(backward=True)
    names = ("q", "k", "v", "log_decay", "gq_logits", "gk_logits")

    def forward(p, x):
        return api.sla_forward(p, *(x[n] for n in names), beta=x["beta"], h0=x["h0"], workspace=ws)[0]

    def backward(p, x):
        return api.sla_backward(p, *(x[n] for n in names), x["dO"], beta=x["beta"], h0=x["h0"], dht=x["dht"], want_dh0=True, workspace=ws)

    ref = [backward(plain, x) for x in layers]
    for p, x in zip(plans, layers):
        forward(p, x)
    got = [backward(p, x) for p, x in list(zip(plans, layers))[::-1]][::-1]
    forward(plans[0], layers[0])
    ws.fill_(255)                                                 # NaN in every value
    got.append(backward(plans[0], layers[0]))
    torch.cuda.synchronize()
    for p in plans + [plain]:
        p.poll()
    for g, r in zip(got, ref + ref[:1]):
        for n, t in r.items():
            if t is not None:
                assert torch.equal(t, g[n]), n
