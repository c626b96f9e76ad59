"""Decode with more steps than the ring of operand blocks holds, several items a CTA with several tokens each, and state widths that end
inside a slice's lines (16, 48, 80, 96, 112 columns of one or two slices): against the oracle, and bit for bit against single tokens."""
import numpy as np
import pytest
import torch

from oracle import sla_oracle as orc
from paper_2602_01744_b200 import api
from paper_2602_01744_b200.inputs import CONFIGS, make_decode_inputs, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", ["retnet", "gla", "gdn"])
@pytest.mark.parametrize("B,H,dk,dv,n,dtype", [(1, 2, 32, 16, 13, "fp32"), (1, 4, 128, 48, 7, "bf16"), (2, 2, 112, 96, 8, "bf16"),
                                               (1, 1, 128, 128, 19, "bf16"), (25, 16, 48, 112, 2, "bf16"), (30, 32, 16, 80, 3, "fp32")])
def test_many_steps_match_the_oracle_and_single_tokens(variant, B, H, dk, dv, n, dtype):
    base = {"retnet": CONFIGS["C0"], "gla": CONFIGS["C1"], "gdn": CONFIGS["C4"]}[variant]
    cfg = small(base, B=B, T=n, H=H, d_k=dk, d_v=dv, dtype=dtype, seed=1970 + dv)
    dec = make_decode_inputs(cfg, B, n, seed=1971)                 # [n, B, H, d]
    tm = lambda t: None if t is None else t.transpose(0, 1).contiguous()
    ld = dec["log_decay"] if variant == "retnet" else tm(dec["log_decay"])
    h0 = torch.randn(B, H, dk, dv, generator=torch.Generator().manual_seed(9)) * 0.1
    plan = api.sla_plan_create(cfg.variant, cfg.dtype, B, 64, H, dk, dv)
    cu = lambda t: None if t is None else t.cuda()
    # a guard row behind the states: a store across the end of the last row would land there
    room = torch.full(((B * H * dk + 1) * dv,), 7.0, device="cuda")
    many = room[:B * H * dk * dv].view(B, H, dk, dv)
    many.copy_(h0)
    o = api.sla_decode_steps(plan, cu(tm(dec["q"])), cu(tm(dec["k"])), cu(tm(dec["v"])), cu(ld), cu(tm(dec["gq_logits"])),
                             cu(tm(dec["gk_logits"])), many, beta=cu(tm(dec["beta"])))
    single, outs = h0.clone().cuda(), []
    for t in range(n):
        at = lambda x: None if x is None else x[t].clone().cuda()
        outs.append(api.sla_decode_step(plan, at(dec["q"]), at(dec["k"]), at(dec["v"]),
                                        cu(ld) if variant == "retnet" else at(dec["log_decay"]), at(dec["gq_logits"]),
                                        at(dec["gk_logits"]), single, beta_t=at(dec["beta"])))
    torch.cuda.synchronize()
    plan.poll()
    assert torch.equal(o, torch.stack(outs, 1)) and torch.equal(many, single)
    assert bool((room[B * H * dk * dv:] == 7.0).all())
    ref = np.ascontiguousarray(h0.double().numpy().copy())
    oref = orc.decode_steps(variant, tm(dec["q"]), tm(dec["k"]), tm(dec["v"]), ld, tm(dec["gq_logits"]), tm(dec["gk_logits"]),
                            ref, beta=tm(dec["beta"]))
    assert gu.rel_l2(o, oref) <= gu.TOL[dtype] and gu.rel_l2(many, ref) <= gu.TOL[dtype]
