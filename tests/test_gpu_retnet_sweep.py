"""The Softmax-RetNet gradient sweep keeps two chunks of input tiles in flight and prepares a chunk while the one before it is worked on:
one to five chunks, full and ragged (every phase of its two buffers and four gate slots), with states at both ends, against the
oracle and bit for bit alike on every run; the decay range it reports."""
import pytest
import torch

from paper_2602_01744_b200 import api
from paper_2602_01744_b200.inputs import CONFIGS, make_inputs, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("T,d", [(1, 128), (64, 128), (65, 128), (128, 64), (190, 128), (256, 128), (257, 64), (320, 128)])
def test_every_number_of_chunks_up_to_five(T, d):
    cfg = small(CONFIGS["R2"], B=2, T=T, H=8, d_k=d, d_v=d, seed=2100 + T)
    x = make_inputs(cfg, with_dO=True, with_h0=True)
    xd = gu.to_dev(x)
    runs = [gu.gpu_training_step(cfg, xd, h0=xd["h0"], dht=xd["dht"], want_dh0=True) for _ in range(4)]
    o, ht, g = runs[0][:3]
    ref = gu.oracle_backward(cfg, x, h0=x["h0"], dht=x["dht"])
    pairs = {n: (g[n], ref[r]) for n, r in gu.GRAD_NAMES.items() if g.get(n) is not None}
    gu.assert_close({n: gu.rel_l2(a, r) for n, (a, r) in pairs.items()},
                    {n: gu.row_err(a, r) for n, (a, r) in pairs.items()}, cfg.dtype, cfg)
    for other in runs[1:]:
        assert torch.equal(o, other[0]) and torch.equal(ht, other[1])
        for n, t in g.items():
            if t is not None:
                assert torch.equal(t, other[2][n]), n


@pytest.mark.parametrize("T,reported", [(64, True), (30, False)])
def test_a_decay_beyond_the_range_of_a_chunk_is_reported(T, reported):
    cfg = small(CONFIGS["R2"], B=1, T=T, H=2, seed=2190)
    x = gu.to_dev(make_inputs(cfg, with_dO=True))
    ld = torch.tensor([-0.1, -2.0], device="cuda")               # -2 a token: -128 over a full chunk, -60 over 30 tokens
    plan = api.sla_plan_create(cfg.variant, cfg.dtype, 1, T, 2, cfg.d_k, cfg.d_v)
    for call in (lambda: api.sla_forward(plan, x["q"], x["k"], x["v"], ld, x["gq_logits"], x["gk_logits"]),
                 lambda: api.sla_backward(plan, x["q"], x["k"], x["v"], ld, x["gq_logits"], x["gk_logits"], x["dO"])):
        call()
        torch.cuda.synchronize()
        if reported:
            with pytest.raises(api.SLAError):
                plan.poll()
        plan.poll()
