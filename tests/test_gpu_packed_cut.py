"""Packed batches whose long sequences are cut into segments (tensor-core Softmax-GLA, -RetNet): outputs, final states and gradients against the
fp64 oracle run sequence by sequence and against the uncut form, which the same calls take with less scratch."""
import numpy as np
import pytest
import torch

from paper_2602_01744_b200 import api
from paper_2602_01744_b200.inputs import CONFIGS, make_inputs, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


# the longest sequence last, first, alone and twice, its last segment short by up to a chunk and of one token; mixed widths; fwd: the forward pass
# is cut, too (with much beside the long sequence only the backward pass is)
@pytest.mark.parametrize("base,lens,H,dk,dv,fwd", [
    ("C2", (64, 1, 2561), 2, 128, 128, True), ("R2", (2700, 130, 63), 2, 128, 128, True), ("C2", (2560, 2497, 65), 1, 64, 128, True),
    ("R2", (2624, ), 1, 128, 64, True), ("C2", (1600, *[64] * 30), 32, 64, 64, False), ("R2", (300, 1601, *[64] * 26), 32, 64, 64, True), ("C2", (2500, 900), 3, 64, 64, True)])
@pytest.mark.parametrize("with_h0", [False, True])
def test_cut_sequences_match_the_oracle_and_the_uncut_form(base, lens, H, dk, dv, fwd, with_h0):
    cu = [0, *np.cumsum(lens).tolist()]
    n, T = len(lens), cu[-1]
    cfg = small(CONFIGS[base], B=1, T=T, H=H, d_k=dk, d_v=dv, seed=2600 + T)
    xh = make_inputs(cfg, with_dO=True)
    if with_h0:
        gen = torch.Generator().manual_seed(T)
        xh["h0"], xh["dht"] = (torch.randn(n, H, dk, dv, generator=gen) * 0.1 for _ in range(2))
    x = gu.to_dev(xh)
    args = (x["q"], x["k"], x["v"], x["log_decay"], x["gq_logits"], x["gk_logits"])
    plan = api.sla_plan_create(cfg.variant, cfg.dtype, 1, T, H, dk, dv, flags=api.SLA_FLAG_SAVE_FOR_BACKWARD)
    plan.set_sequences(cu)

    def step(fwd_ws, bwd_ws):
        ht = torch.full((n, H, dk, dv), float("nan"), device="cuda")
        o, _ = api.sla_forward(plan, *args, h0=x.get("h0"), ht=ht, workspace=fwd_ws)
        launches = [plan.last_launch_count]
        g = api.sla_backward(plan, *args, x["dO"], h0=x.get("h0"), dht=x.get("dht"), want_dh0=True, workspace=bwd_ws)
        return {"o": o, "ht": ht, **{k: t for k, t in g.items() if t is not None}}, launches + [plan.last_launch_count]

    ws, ws2 = plan.workspace(backward=True), plan.workspace(backward=True)
    uncut = torch.empty(sum(-(-m // 64) + 1 for m in lens) * H * (32 << 10) + 2 * -(-T * H * 4 // 256) * 256, dtype=torch.uint8, device="cuda")
    assert uncut.numel() < ws.numel()
    got, launches = step(ws, ws)
    assert launches == [3 if fwd else 1, 4]
    again, launches = step(ws, ws2)
    assert launches == ([3, 7] if fwd else [1, 5])                             # other workspace: recomputed, the same bits
    whole, launches = step(uncut, uncut)
    assert launches == [1, 2]
    mixed, launches = step(uncut, ws)                      # what the other form left is not taken
    assert launches == [1, 7 if fwd else 5]
    torch.cuda.synchronize()
    plan.poll()
    refs = {}
    for s in range(n):
        a, b = cu[s], cu[s + 1]
        c1 = small(cfg, T=b - a)
        xs = {k: t if t is None or t.dim() == 1 else t[s:s + 1] if k in ("h0", "dht") else t[:, a:b].contiguous() for k, t in xh.items()}
        oref, htref = gu.oracle_forward(c1, xs, h0=xs.get("h0"))
        ref = gu.oracle_backward(c1, xs, h0=xs.get("h0"), dht=xs.get("dht"))
        for k, t in {"o": oref, "ht": htref, **{k: ref[r] for k, r in gu.GRAD_NAMES.items() if k in got}}.items():
            refs.setdefault(k, []).append(t)
    refs = {k: np.concatenate(v, axis=0 if k in ("ht", "dh0") else 1) for k, v in refs.items()}
    for res in (got, whole):
        gu.assert_close({k: gu.rel_l2(res[k], r) for k, r in refs.items()}, {k: gu.row_err(res[k], r) for k, r in refs.items()}, cfg.dtype, cfg)
    for k, t in got.items():
        assert torch.equal(t, again[k]), k
        assert k in ("o", "ht") or torch.equal(t, mixed[k]), k


@pytest.mark.parametrize("base,lens,d,launches", [
    ("C2", (2560, *[64] * 170), 64, [1, 4, 5]), ("R2", (2560, *[64] * 170), 64, [1, 4, 5]), ("C2", (6400, *[64] * 130), 64, [3, 4, 7]),
    ("C2", (2560, *[64] * 60), 128, [1, 4, 5])])
def test_large_batches_give_the_uncut_form_s_gradients(base, lens, d, launches):
    """Cut and uncut passes read one another's state images: pairs of 64-wide heads in both forms, single heads whole and pairs cut, wide heads."""
    cu, n, H = [0, *np.cumsum(lens).tolist()], len(lens), 32
    cfg = small(CONFIGS[base], B=1, T=cu[-1], H=H, d_k=d, d_v=d, seed=2800 + len(lens))
    x = gu.to_dev(make_inputs(cfg, with_dO=True))
    gen = torch.Generator(device="cuda").manual_seed(7)
    h0, dht = (torch.randn(n, H, d, d, generator=gen, device="cuda") * 0.1 for _ in range(2))
    args = (x["q"], x["k"], x["v"], x["log_decay"], x["gq_logits"], x["gk_logits"])
    plan = api.sla_plan_create(cfg.variant, cfg.dtype, 1, cfg.T, H, d, d, flags=api.SLA_FLAG_SAVE_FOR_BACKWARD)
    plan.set_sequences(cu)
    ws, ws2 = plan.workspace(backward=True), plan.workspace(backward=True)
    whole = torch.empty(sum(-(-m // 64) + 1 for m in lens) * H * (32 << 10) + 2 * -(-cfg.T * H * 4 // 256) * 256, dtype=torch.uint8, device="cuda")

    def step(fwd_ws, bwd_ws, start, end):
        o, _ = api.sla_forward(plan, *args, h0=start, ht=end, workspace=fwd_ws)
        count = [plan.last_launch_count]
        g = api.sla_backward(plan, *args, x["dO"], h0=start, dht=dht, want_dh0=True, workspace=bwd_ws)
        return {"o": o, "ht": end, **{k: t for k, t in g.items() if t is not None}}, count + [plan.last_launch_count]

    ref, count = step(whole, whole, h0, torch.empty_like(h0))
    assert count == [1, 2]
    runs = [step(ws, ws, h0, torch.empty_like(h0)), step(ws, ws2, h0, torch.empty_like(h0))]
    assert [c for _, c in runs] == [launches[:2], [launches[0], launches[2]]]
    torch.cuda.synchronize()
    plan.poll()
    for k, t in runs[0][0].items():
        assert torch.equal(t, runs[1][0][k]), k
        assert gu.rel_l2(t, ref[k].double().cpu().numpy()) <= 1e-2, k


def test_short_or_balanced_batches_are_not_cut():
    for lens, H in [((900, 64, 64), 2), ((1024,) * 20, 16)]:
        plan = api.sla_plan_create("gla", "bf16", 1, sum(lens), H, 128, 128)
        plan.set_sequences([0, *np.cumsum(lens).tolist()])
        assert plan.forward_workspace_bytes == 0


def test_states_in_one_buffer():
    lens, H = (64, 2561), 2
    cu = [0, *np.cumsum(lens).tolist()]
    cfg = small(CONFIGS["C2"], B=1, T=cu[-1], H=H, seed=2700)
    x = gu.to_dev(make_inputs(cfg, with_dO=True))
    args = (x["q"], x["k"], x["v"], x["log_decay"], x["gq_logits"], x["gk_logits"])
    h0 = torch.randn(2, H, 128, 128, generator=torch.Generator(device="cuda").manual_seed(5), device="cuda") * 0.1
    plan = api.sla_plan_create(cfg.variant, cfg.dtype, 1, cfg.T, H, 128, 128)
    plan.set_sequences(cu)
    ht = torch.empty_like(h0)
    o, _ = api.sla_forward(plan, *args, h0=h0, ht=ht)
    assert plan.last_launch_count == 3
    state = h0.clone()
    o2, _ = api.sla_forward(plan, *args, h0=state, ht=state)
    assert plan.last_launch_count == 1
    torch.cuda.synchronize()
    plan.poll()
    assert gu.rel_l2(o2, o.double().cpu().numpy()) <= 1e-2 and gu.rel_l2(state, ht.double().cpu().numpy()) <= 1e-2


@pytest.mark.parametrize("base", ["C2", "R2"])
def test_state_gradients_in_one_buffer(base):
    """dh0 in dht's buffer: a segment may write its sequence's dh0 before the last one has read dht, so the backward pass runs uncut."""
    lens, H = (64, 2561), 2
    cu = [0, *np.cumsum(lens).tolist()]
    cfg = small(CONFIGS[base], B=1, T=cu[-1], H=H, seed=2710)
    x = gu.to_dev(make_inputs(cfg, with_dO=True))
    args = (x["q"], x["k"], x["v"], x["log_decay"], x["gq_logits"], x["gk_logits"])
    dht = torch.randn(2, H, 128, 128, generator=torch.Generator(device="cuda").manual_seed(6), device="cuda") * 0.1
    plan = api.sla_plan_create(cfg.variant, cfg.dtype, 1, cfg.T, H, 128, 128)
    plan.set_sequences(cu)
    ws = plan.workspace(backward=True)
    g = api.sla_backward(plan, *args, x["dO"], dht=dht, want_dh0=True, workspace=ws)
    assert plan.last_launch_count == 7
    state = dht.clone()
    out = {n: None if t is None else torch.empty_like(t) for n, t in g.items()}
    out["dh0"] = state
    api.sla_backward(plan, *args, x["dO"], dht=state, workspace=ws, out=out)
    assert plan.last_launch_count == 3
    whole = torch.empty(sum(-(-m // 64) + 1 for m in lens) * H * (32 << 10) + 2 * -(-cfg.T * H * 4 // 256) * 256, dtype=torch.uint8, device="cuda")
    ref = api.sla_backward(plan, *args, x["dO"], dht=dht, want_dh0=True, workspace=whole)
    assert plan.last_launch_count == 3
    torch.cuda.synchronize()
    plan.poll()
    for n, t in ref.items():
        if t is not None:
            assert torch.equal(t, out[n]), n
            assert gu.rel_l2(g[n], t.double().cpu().numpy()) <= 1e-2, n


@pytest.mark.parametrize("flags", [0, api.SLA_FLAG_SAVE_FOR_BACKWARD])
def test_calls_without_a_workspace_run_uncut_where_memory_is_short(monkeypatch, flags):
    lens, H = (64, 2561), 2
    cu = [0, *np.cumsum(lens).tolist()]
    cfg = small(CONFIGS["C2"], B=1, T=cu[-1], H=H, seed=2720)
    x = gu.to_dev(make_inputs(cfg, with_dO=True))
    args = (x["q"], x["k"], x["v"], x["log_decay"], x["gq_logits"], x["gk_logits"])
    plan = api.sla_plan_create(cfg.variant, cfg.dtype, 1, cfg.T, H, 128, 128, flags=flags)
    plan.set_sequences(cu)
    calls = [lambda: api.sla_forward(plan, *args)[0], lambda: api.sla_backward(plan, *args, x["dO"])["dq"]]
    cut = [(c(), plan.last_launch_count) for c in calls]
    assert [n for _, n in cut] == [3, 7]
    real = torch.empty

    def short(*size, **kw):
        if kw.get("dtype") == torch.uint8 and size[0] in (plan.forward_workspace_bytes, plan.backward_workspace_bytes):
            raise torch.OutOfMemoryError("short")
        return real(*size, **kw)

    monkeypatch.setattr(torch, "empty", short)
    uncut = [(c(), plan.last_launch_count) for c in calls]
    assert [n for _, n in uncut] == [1, 3]
    torch.cuda.synchronize()
    plan.poll()
    for (a, _), (b, _) in zip(cut, uncut):
        assert gu.rel_l2(a, b.double().cpu().numpy()) <= 1e-2
