"""Decode in column slices: state widths that fill one slice, part of one, or two; key widths below 128; more items than the
persistent CTAs; one and several tokens a call (which run in slices of different width) against the oracle, bit for bit alike."""
import numpy as np
import pytest
import torch

from oracle import sla_oracle as orc
from paper_2602_01744_b200 import api
from paper_2602_01744_b200.inputs import CONFIGS, make_decode_inputs, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", ["retnet", "gla", "gdn"])
@pytest.mark.parametrize("B,H,dk,dv,dtype", [(1, 4, 16, 16, "fp32"), (2, 4, 80, 64, "bf16"), (2, 8, 128, 80, "fp32"),
                                             (1, 1, 64, 112, "bf16"), (40, 16, 64, 128, "bf16")])
def test_slices_match_the_oracle_and_one_another(variant, B, H, dk, dv, dtype):
    n = 3
    base = {"retnet": CONFIGS["C0"], "gla": CONFIGS["C1"], "gdn": CONFIGS["C4"]}[variant]
    cfg = small(base, B=B, T=n, H=H, d_k=dk, d_v=dv, dtype=dtype, seed=970 + dv)
    dec = make_decode_inputs(cfg, B, n, seed=971)                  # [n, B, H, d]
    tm = lambda t: None if t is None else t.transpose(0, 1).contiguous()
    ld = dec["log_decay"] if variant == "retnet" else tm(dec["log_decay"])
    h0 = torch.randn(B, H, dk, dv, generator=torch.Generator().manual_seed(9)) * 0.1
    plan = api.sla_plan_create(cfg.variant, cfg.dtype, B, 64, H, dk, dv)
    cu = lambda t: None if t is None else t.cuda()
    many = h0.clone().cuda()
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
    ref = np.ascontiguousarray(h0.double().numpy().copy())
    oref = orc.decode_steps(variant, tm(dec["q"]), tm(dec["k"]), tm(dec["v"]), ld, tm(dec["gq_logits"]), tm(dec["gk_logits"]),
                            ref, beta=tm(dec["beta"]))
    assert gu.rel_l2(o, oref) <= gu.TOL[dtype] and gu.rel_l2(many, ref) <= gu.TOL[dtype]
