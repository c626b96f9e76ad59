"""The native marshalling of the decode calls against the Python path: the same bits, outputs handed in or allocated, on a stream of its own
and from several threads, and the same refusals."""
import threading

import pytest
import torch

from paper_2602_01744_b200 import api

pytestmark = pytest.mark.gpu


def _inputs(variant, n, dtype, seed, B=3, H=4, d=32):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")
    tok = (B, n, H) if n else (B, H)
    ld = -torch.rand(H if variant == "retnet" else tok + ((d,) if variant == "gla" else ()), generator=g, device="cuda")
    kw = {("beta" if n else "beta_t"): torch.rand(tok, generator=g, device="cuda")} if variant == "gdn" else {}
    return [r(*tok, d).to(dtype), r(*tok, d).to(dtype), r(*tok, d).to(dtype), ld, r(*tok), r(*tok)], kw, r(B, H, d, d)


@pytest.mark.parametrize("variant", ["retnet", "gla", "gdn"])
@pytest.mark.parametrize("n,dtype", [(0, "bf16"), (3, "fp32")])
def test_the_two_paths_give_the_same_bits(variant, n, dtype, monkeypatch):
    assert api.lib() and api._fast is not None, "the native marshalling is not built"
    plan = api.sla_plan_create(variant, dtype, 3, max(n, 1), 4, 32, 32)
    step = api.sla_decode_steps if n else api.sla_decode_step
    args, kw, state = _inputs(variant, n, plan.io_torch, 5)
    out = "o" if n else "o_t"
    states = [state.clone() for _ in range(4)]
    o = [step(plan, *args, states[0], **kw)]
    given = torch.empty_like(o[0])
    o.append(step(plan, *args, states[1], **kw, **{out: given}))
    assert o[1] is given and o[0].dtype == plan.io_torch
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        o.append(step(plan, *args, states[2], **kw))
    torch.cuda.current_stream().wait_stream(side)
    monkeypatch.setattr(api, "_fast", None)
    o.append(step(plan, *args, states[3], **kw))
    torch.cuda.synchronize()
    plan.poll()
    for a, s in zip(o, states):
        assert torch.equal(a, o[3]) and torch.equal(s, states[3])


def test_refusals_are_the_same(monkeypatch):
    plan = api.sla_plan_create("gla", "bf16", 3, 1, 4, 32, 32)
    args, kw, state = _inputs("gla", 0, torch.bfloat16, 6)
    fast = api._fast
    for f in (fast, None):
        monkeypatch.setattr(api, "_fast", f)
        with pytest.raises(AssertionError):                                   # not contiguous
            api.sla_decode_step(plan, args[0].transpose(0, 1).contiguous().transpose(0, 1), *args[1:], state)
        with pytest.raises(AssertionError):                                   # not on the GPU
            api.sla_decode_step(plan, *args, state.cpu())
        with pytest.raises(api.SLAError) as e:                                # refused by the library: no log-decay
            api.sla_decode_step(plan, *args[:3], None, *args[4:], state)
        assert e.value.status == 1
        with pytest.raises(api.SLAError):                                     # misaligned state
            api.sla_decode_step(plan, *args, torch.empty(state.numel() + 1, device="cuda")[1:].view(state.shape))


def test_threads_with_states_of_their_own():
    plans, got = [api.sla_plan_create("gdn", "fp32", 3, 1, 4, 32, 32) for _ in range(4)], [None] * 4
    data = [_inputs("gdn", 0, torch.float32, 7 + i) for i in range(4)]
    ref = []
    for p, (args, kw, state) in zip(plans, data):
        s = state.clone()
        for _ in range(20):
            o = api.sla_decode_step(p, *args, s, **kw)
        ref.append((o, s))
    torch.cuda.synchronize()

    def work(i):
        args, kw, state = data[i]
        with torch.cuda.stream(torch.cuda.Stream()):
            for _ in range(20):
                o = api.sla_decode_step(plans[i], *args, state, **kw)
            torch.cuda.current_stream().synchronize()
        got[i] = (o, state)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for (o, s), (a, b) in zip(ref, got):
        assert torch.equal(o, a) and torch.equal(s, b)
