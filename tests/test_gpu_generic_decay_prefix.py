"""The cumulative log-decay of the fp32 kernels next to a token that forgets nearly everything: the token before it keeps its precision."""
import numpy as np
import pytest
import torch

from paper_2602_01744_b200 import api
from oracle import sla_oracle as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunk", [16, 64])
@pytest.mark.parametrize("p", [1, 7, 15])
def test_the_token_before_a_strong_decay(p, chunk):
    """beta ~ 0: a token's output is e^b q h0, d_k products whose factors each carry a few roundings: at most (d_k + 8) 2^-24 of sum |q h0| e^b."""
    B, T, H, d = 4, 40, 16, 16
    gen = torch.Generator().manual_seed(31 + p)
    r = lambda *s: torch.randn(*s, generator=gen)
    q, k, v = r(B, T, H, d), torch.nn.functional.normalize(r(B, T, H, d), dim=-1), r(B, T, H, d)
    decay = -0.01 * torch.rand(B, T, H, generator=gen)
    decay[:, p] = -70.0
    beta, lq, lk, h0 = torch.full((B, T, H), 1e-8), r(B, T, H), r(B, T, H), r(B, H, d, d)
    plan = api.sla_plan_create("gdn", "fp32", B, T, H, d, d, chunk)
    o, _ = api.sla_forward(plan, *(x.cuda() for x in (q, k, v, decay, lq, lk)), beta=beta.cuda(), h0=h0.cuda())
    torch.cuda.synchronize()
    plan.poll()
    ref, _ = orc.forward("gdn", q, k, v, decay, lq, lk, beta=beta, h0=h0)
    gate = torch.softmax(lq.double(), -1)[:, p - 1, :, None]
    b = decay.double()[:, :p].sum(1)[..., None]
    size = torch.einsum("bhk,bhkv->bhv", q.double()[:, p - 1].abs(), h0.double().abs()) * gate * b.exp()
    err = np.abs(o[:, p - 1].double().cpu().numpy() - ref[:, p - 1]) / size.numpy()
    assert err.max() <= (d + 8) * 2.0 ** -24
