"""64-wide heads, more of them than SMs: two heads of a pair share a CTA (Softmax-GLA and -RetNet).  Against the oracle, with states at both
ends, regular and packed; the recomputing backward and single heads (few enough to run on their own) give the same gradients."""
import pytest
import torch

from oracle import sla_oracle as orc
from paper_2602_01744_b200 import api
from paper_2602_01744_b200.inputs import CONFIGS, make_inputs, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base", ["C2", "R2"])
@pytest.mark.parametrize("B,T,H", [(10, 130, 16), (75, 65, 2), (26, 5, 6), (5, 320, 32), (38, 64, 4)])
def test_pairs_match_the_oracle(base, B, T, H):
    cfg = small(CONFIGS[base], B=B, T=T, H=H, d_k=64, d_v=64, seed=2300 + T)
    x = make_inputs(cfg, with_dO=True, with_h0=True)
    xd = gu.to_dev(x)
    kw = dict(h0=xd["h0"], dht=xd["dht"], want_dh0=True)
    o, ht, g, plan, ws, lf, lb = gu.gpu_training_step(cfg, xd, **kw)
    assert (lf, lb) == (1, 2)
    oref, htref = gu.oracle_forward(cfg, x, h0=x["h0"])
    ref = gu.oracle_backward(cfg, x, h0=x["h0"], dht=x["dht"])
    pairs = {"o": (o, oref), "ht": (ht, htref)}
    pairs.update({n: (g[n], ref[r]) for n, r in gu.GRAD_NAMES.items() if g.get(n) is not None})
    gu.assert_close({n: gu.rel_l2(a, r) for n, (a, r) in pairs.items()},
                    {n: gu.row_err(a, r) for n, (a, r) in pairs.items()}, cfg.dtype, cfg)
    # the recomputing backward, and the step over and over, give the same bits
    g2, plan2 = gu.gpu_backward(cfg, xd, **kw)
    assert plan2.last_launch_count == 3
    again = gu.gpu_training_step(cfg, xd, **kw)
    assert torch.equal(o, again[0]) and torch.equal(ht, again[1])
    for n, t in g.items():
        if t is not None:
            assert torch.equal(t, g2[n]) and torch.equal(t, again[2][n]), n
    # without states at the ends (none read, none left)
    plain = api.sla_plan_create(cfg.variant, cfg.dtype, B, T, H, 64, 64)
    args = (xd["q"], xd["k"], xd["v"], xd["log_decay"], xd["gq_logits"], xd["gk_logits"])
    o0, _ = api.sla_forward(plain, *args)
    g0 = api.sla_backward(plain, *args, xd["dO"])
    torch.cuda.synchronize()
    plain.poll()
    ref0 = gu.oracle_backward(cfg, x)
    assert gu.rel_l2(o0, gu.oracle_forward(cfg, x)[0]) <= 1e-2
    assert max(gu.rel_l2(g0[n], ref0[r]) for n, r in gu.GRAD_NAMES.items() if g0.get(n) is not None) <= 1e-2


@pytest.mark.parametrize("base", ["C2", "R2"])
def test_packed_pairs_match_sequences_run_alone(base):
    """Thirty-six sequences of 16 heads (more chunks an SM than the longest sequence has: paired) against each sequence as a call of its
    own (16 heads: single)."""
    lens = [1, 63, 64, 65, 300, 130, 2, 128, 129, 17, 190, 64] * 3
    H, cu = 16, [0]
    for n in lens:
        cu.append(cu[-1] + n)
    cfg = small(CONFIGS[base], B=1, T=cu[-1], H=H, d_k=64, d_v=64, seed=2390)
    x = gu.to_dev(make_inputs(cfg, with_dO=True))
    gen = torch.Generator(device="cuda").manual_seed(3)
    h0, dht = (torch.randn(len(lens), H, 64, 64, generator=gen, device="cuda") * 0.1 for _ in range(2))
    names = ("q", "k", "v", "log_decay", "gq_logits", "gk_logits")
    plan = api.sla_plan_create(cfg.variant, cfg.dtype, 1, cfg.T, H, 64, 64, flags=api.SLA_FLAG_SAVE_FOR_BACKWARD)
    plan.set_sequences(cu)
    ws, ht = plan.workspace(backward=True), torch.empty_like(h0)
    o, _ = api.sla_forward(plan, *(x[n] for n in names), h0=h0, ht=ht, workspace=ws)
    g = api.sla_backward(plan, *(x[n] for n in names), x["dO"], h0=h0, dht=dht, want_dh0=True, workspace=ws)
    torch.cuda.synchronize()
    plan.poll()
    for s, (a, b) in enumerate(zip(cu, cu[1:])):
        cut = lambda t: t if t is None or t.dim() == 1 else t[:, a:b].contiguous()
        p1 = api.sla_plan_create(cfg.variant, cfg.dtype, 1, b - a, H, 64, 64)
        args = [cut(x[n]) for n in names]
        ht1 = torch.empty_like(h0[:1])
        o1, _ = api.sla_forward(p1, *args, h0=h0[s:s + 1], ht=ht1)
        g1 = api.sla_backward(p1, *args, cut(x["dO"]), h0=h0[s:s + 1], dht=dht[s:s + 1], want_dh0=True)
        pairs = [(o[:, a:b], o1), (ht[s:s + 1], ht1), (g["dh0"][s:s + 1], g1["dh0"])]
        pairs += [(g[n][:, a:b], t) for n, t in g1.items() if t is not None and n != "dh0"]
        for got, want in pairs:      # the same products in the same precision, sums over a head's 64 features in another order
            assert gu.rel_l2(got, want.double().cpu().numpy()) <= 2e-3, (s, got.shape)
