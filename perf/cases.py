"""Performance cases of the Softmax-Linear-Attention library: what a serving loop and a training step have it do.

A case is a plain dict.  `kind` says which calls one pass makes:

  decode   sla_decode_step(s) on a caller-held state: a serving loop (n tokens per sequence per call)
  prefill  sla_forward with the final state: a prompt, or the continuation of one (h0) - inference, nothing is saved
  train    sla_forward + sla_backward on a SLA_FLAG_SAVE_FOR_BACKWARD plan: the layer inside a training step
  packed   the same on one row of packed variable-length sequences (sla_plan_set_sequences)
  layer    a whole training step around the layer: feature map (GDN), gate scores, layer, output projection, and back

Inputs follow the distributions of `paper_2602_01744_b200.inputs`, drawn on the GPU.
"""
import random

import torch

from paper_2602_01744_b200 import api


def _case(name, kind, variant, B, T, H, dk, dv, dtype="bf16", n=1, h0=False, n_seq=0):
    c = dict(kind=kind, variant=variant, dtype=dtype, B=B, T=T, H=H, dk=dk, dv=dv, n=n, h0=h0, n_seq=n_seq)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one user's token stream, one token a call: launch and latency
        _case("decode_gla_one", "decode", "gla", 1, 1, 16, 128, 128),
        # a serving batch of 64 streams, one token each: 64 MiB of state read and written
        _case("decode_gla_batch", "decode", "gla", 64, 1, 16, 128, 128),
        # eight speculated tokens verified for each of 16 streams in one call
        _case("decode_gdn_verify", "decode", "gdn", 16, 1, 16, 128, 128, n=8),
        # a batch of short prompts (the C1 shape)
        _case("prefill_gla", "prefill", "gla", 4, 2048, 8, 128, 128),
        # one long document (the C3 shape)
        _case("prefill_gla_long", "prefill", "gla", 1, 65536, 16, 128, 128),
        # prompts of a length that is no multiple of the chunk, continued from an earlier state
        _case("prefill_gdn_ragged", "prefill", "gdn", 3, 2500, 16, 128, 128, h0=True),
        # the layer of a training step at the paper's training length: the three instantiations (C2, R2, C4 shapes)
        _case("train_gla", "train", "gla", 8, 4096, 16, 128, 128),
        _case("train_retnet", "train", "retnet", 8, 4096, 16, 128, 128),
        _case("train_gdn", "train", "gdn", 4, 4096, 16, 128, 128),
        # training data packed to a token budget, more and narrower heads
        _case("train_packed_narrow", "packed", "gla", 1, 16384, 32, 64, 64, n_seq=17),
        # a whole Gated-DeltaNet layer step: feature map, gate scores, layer, W^O, and the way back
        _case("layer_gdn", "layer", "gdn", 2, 2048, 16, 128, 128),
        # the precision path: fp32 in and out (C0's heads at a length a numerical check would use)
        _case("train_fp32", "train", "retnet", 2, 1000, 4, 64, 64, dtype="fp32"),
    ]


def _log_int(rng, lo, hi):
    """An integer in lo .. hi, uniform in its logarithm."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["decode", "decode", "prefill", "prefill", "train", "train", "train", "packed", "layer", "fp32"])
    variant = rng.choice(["gla", "retnet", "gdn"])
    if kind == "fp32":
        d = rng.choice([32, 64, 64, 96])
        return _case(None, "train", variant, _log_int(rng, 1, 4), _log_int(rng, 60, 1000), rng.choice([2, 4]), d, d,
                     dtype="fp32", h0=rng.random() < 0.3)
    H = rng.choice([4, 8, 8, 16, 16, 16, 32])
    dk, dv = rng.choice([(128, 128), (128, 128), (128, 128), (64, 64), (64, 128)])
    if kind == "decode":
        B = _log_int(rng, 1, 1024 // H)
        return _case(None, kind, variant, B, 1, H, dk, dv, n=rng.choice([1, 1, 1, 2, 4, 5, 8]))
    # tokens x heads of a pass: the GDN layer does the most work per pair
    most = 2 ** 18 if variant == "gdn" or (dk, dv) != (128, 128) else 2 ** 19
    if kind == "layer":
        most = 2 ** 16
    pairs = _log_int(rng, most // 32, most)
    if kind == "packed":
        T = max(512, pairs // H)
        return _case(None, kind, variant, 1, T, H, dk, dv, n_seq=rng.randint(3, 24))
    B = 1 if kind == "prefill" and rng.random() < 0.4 else _log_int(rng, 1, 8)
    T = max(64, pairs // (H * B))
    if rng.random() < 0.5:
        T -= rng.randint(1, 63)
    if T * B * H < 1024:
        T = 1024 // (B * H) + 64
    if kind != "prefill":
        T = min(T, 8192)
    return _case(None, kind, variant, B, T, H, dk, dv, h0=kind == "prefill" and rng.random() < 0.4)


def _lengths(case):
    """The cut of a packed row: n_seq lengths of which none is empty and the longest takes a good part of the row."""
    r = random.Random(1000003 * case["T"] + case["n_seq"])
    w = [r.expovariate(1.0) + 0.02 for _ in range(case["n_seq"])]
    cuts, acc = [0], 0.0
    for x in w[:-1]:
        acc += x
        cuts.append(max(cuts[-1] + 1, int(case["T"] * acc / sum(w))))
    return cuts + [case["T"]]


def _decay(variant, gen, shape, dk):
    if variant == "retnet":
        h = torch.arange(shape[-1], dtype=torch.float64, device="cuda")
        return torch.log(1.0 - torch.pow(2.0, -5.0 - h)).float()
    full = shape + (dk,) if variant == "gla" else shape
    return torch.nn.functional.logsigmoid(torch.randn(full, generator=gen, device="cuda")) / 16.0


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    io = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    kind, variant, H, dk, dv = case["kind"], case["variant"], case["H"], case["dk"], case["dv"]

    def randn(*shape):
        return torch.randn(shape, generator=gen, device="cuda")

    B, T = case["B"], case["T"]
    if kind == "decode":
        T = case["n"]
    tok = (B, T, H) if kind != "decode" or case["n"] > 1 else (B, H)
    s = dict(case=case, plan=api.sla_plan_create(variant, case["dtype"], B, T, H, dk, dv,
                                                 flags=0 if kind in ("decode", "prefill") else api.SLA_FLAG_SAVE_FOR_BACKWARD))
    plan = s["plan"]
    if kind == "packed":
        plan.set_sequences(_lengths(case))
    s["decay"] = _decay(variant, gen, tok, dk)
    s["beta"] = torch.sigmoid(randn(*tok)) if variant == "gdn" else None
    if kind == "layer":
        # activations the input projections leave, the feature map's taps, the gate projections and W^O
        for x, d in (("q", dk), ("k", dk), ("v", dv)):
            s["x_" + x] = randn(*tok, d).to(io)
            s["taps_" + x] = randn(H * d, 4) * 0.5
        s["w_gq"], s["w_gk"] = randn(dk, H), randn(dk, H)
        s["w_o"] = (randn(H * dv, H * dv) / (H * dv) ** 0.5).to(io)
        s["dy"] = randn(B, T, H * dv).to(io)
        if variant != "gdn":
            s["x_q"], s["x_k"], s["x_v"] = (s["x_q"] / dk ** 0.5).to(io), (s["x_k"] / dk ** 0.5).to(io), (s["x_v"] / dv ** 0.5).to(io)
    else:
        s["q"] = (randn(*tok, dk) / dk ** 0.5).to(io)
        k = randn(*tok, dk) / dk ** 0.5
        s["k"] = (k / k.norm(dim=-1, keepdim=True) if variant == "gdn" else k).to(io)
        s["v"] = (randn(*tok, dv) / dv ** 0.5).to(io)
        s["lq"], s["lk"] = randn(*tok), randn(*tok)
    if kind == "decode":
        s["state"] = randn(B, H, dk, dv) * 0.1
        return s
    s["h0"] = randn(B, H, dk, dv) * 0.1 if case["h0"] else None
    s["ht"] = torch.empty((case["n_seq"] or B, H, dk, dv), dtype=torch.float32, device="cuda")
    if kind in ("train", "packed"):
        s["dO"] = randn(*tok, dv).to(io)
    s["ws"] = plan.workspace(backward=kind != "prefill")
    return s


def _run_layer(s):
    plan, gdn = s["plan"], s["case"]["variant"] == "gdn"
    q, k, v = s["x_q"], s["x_k"], s["x_v"]
    if gdn:
        q = api.sla_shortconv_forward(plan, q, s["taps_q"], True)
        k = api.sla_shortconv_forward(plan, k, s["taps_k"], True)
        v = api.sla_shortconv_forward(plan, v, s["taps_v"], False)
    lq, lk = api.sla_gate_scores_forward(plan, q, k, s["w_gq"], s["w_gk"])
    o, _ = api.sla_forward(plan, q, k, v, s["decay"], lq, lk, beta=s["beta"], workspace=s["ws"])
    y = api.sla_out_proj_forward(plan, o, s["w_o"])
    d_o, dw_o = api.sla_out_proj_backward(plan, o, s["w_o"], s["dy"])
    g = api.sla_backward(plan, q, k, v, s["decay"], lq, lk, d_o, beta=s["beta"], workspace=s["ws"])
    dw_gq, dw_gk = api.sla_gate_scores_backward(plan, q, k, s["w_gq"], s["w_gk"], g["dgq_logits"], g["dgk_logits"],
                                                g["dq"], g["dk"])
    out = dict(y=y, dw_o=dw_o, dw_gq=dw_gq, dw_gk=dw_gk, dlog_decay=g["dlog_decay"], dbeta=g["dbeta"])
    for n, x in (("q", g["dq"]), ("k", g["dk"]), ("v", g["dv"])):
        if gdn:
            out["dx_" + n], out["dtaps_" + n] = api.sla_shortconv_backward(plan, s["x_" + n], s["taps_" + n], x, n != "v")
        else:
            out["dx_" + n] = x
    return out


def run(s):
    kind, plan = s["case"]["kind"], s["plan"]
    if kind == "layer":
        return _run_layer(s)
    args = (s["q"], s["k"], s["v"], s["decay"], s["lq"], s["lk"])
    if kind == "decode":
        step = api.sla_decode_step if s["q"].dim() == 3 else api.sla_decode_steps
        if s["q"].dim() == 3:
            o = step(plan, *args, s["state"], beta_t=s["beta"])
        else:
            o = step(plan, *args, s["state"], beta=s["beta"])
        return dict(o=o, state=s["state"])
    o, ht = api.sla_forward(plan, *args, beta=s["beta"], h0=s["h0"], ht=s["ht"], workspace=s["ws"])
    if kind == "prefill":
        return dict(o=o, ht=ht)
    g = api.sla_backward(plan, *args, s["dO"], beta=s["beta"], h0=s["h0"], workspace=s["ws"])
    return dict(o=o, ht=ht, **g)


def work(case):
    """Bytes and operations one pass cannot do without: inputs once, outputs once; the recurrence's own arithmetic."""
    kind, variant, H, dk, dv = case["kind"], case["variant"], case["H"], case["dk"], case["dv"]
    e = 2 if case["dtype"] == "bf16" else 4
    decay = dict(retnet=0, gla=4 * dk, gdn=8)[variant]          # log-decay (and beta) of a (token, head) pair
    pairs = case["B"] * H * (case["n"] if kind == "decode" else case["T"])
    fwd_b = e * (2 * dk + 2 * dv) + decay + 8                    # q, k, v, o, decay, two logits
    bwd_b = e * (4 * dk + 3 * dv) + 2 * decay + 16               # q, k, v, dO, dq, dk, dv, decay and logits with gradients
    fwd_f, bwd_f = (6 if variant == "gdn" else 4) * dk * dv, (16 if variant == "gdn" else 10) * dk * dv
    state = 4 * dk * dv * H
    if kind == "decode":
        return dict(bytes=pairs * fwd_b + 2 * case["B"] * state, flops=pairs * fwd_f)
    if kind == "prefill":
        return dict(bytes=pairs * fwd_b + case["B"] * state * (2 if case["h0"] else 1), flops=pairs * fwd_f)
    total = dict(bytes=pairs * (fwd_b + bwd_b) + (case["n_seq"] or case["B"]) * state, flops=pairs * (fwd_f + bwd_f))
    if kind == "layer":
        tokens, Dv = case["B"] * case["T"], H * dv
        conv = pairs * e * 2 * (2 * dk + dv) if variant == "gdn" else 0
        total["bytes"] += tokens * Dv * e * 4 + Dv * Dv * (e + 4) + conv
        total["flops"] += 6 * tokens * Dv * Dv + pairs * 8 * dk
    return total


def tolerance(case):
    # the tensor-core path against the fp32 kernels on the same bits: 3.5e-3 .. 5e-3 per tensor, single values up to 0.24
    # (rows of a few tokens that cancel); the fp32 kernels with chunks of 16 against chunks of 64: 6e-7, values to 7e-6
    return {"rel": 1.5e-2, "max": 0.6} if case["dtype"] == "bf16" else {"rel": 1e-5, "max": 2e-4}


# ---------------------------------------------------------------------------------------------------------------
# the same results in 64 bits, from the equations of the layer alone (chunks of 64 tokens, reverse pass by autograd)

def _exact_sequence(variant, q, k, v, g, beta, state):
    """One batch of equally long sequences, [B, H, T, d]: q and k (GDN: q and v) already carry their gates."""
    outs = []
    n = q.shape[2]
    parts = [x.split(64, 2) if x is not None else None for x in (q, k, v, g, beta)]
    for i in range((n + 63) // 64):
        qc, kc, vc, gc = (p[i] for p in parts[:4])
        b = gc.cumsum(2)                                     # [B, H, C, d_k or 1]
        last = b[:, :, -1:]
        if variant == "gdn":
            ratio = torch.exp((b - b.transpose(2, 3)).tril())            # e^{b_i - b_j} for j <= i
            low = (parts[4][i] * (kc @ kc.transpose(2, 3)) * ratio).tril(-1)
            rhs = parts[4][i] * (vc - torch.exp(b) * (kc @ state))
            u = torch.linalg.solve_triangular(low, rhs, upper=False, unitriangular=True)
            outs.append((qc * torch.exp(b)) @ state + ((qc @ kc.transpose(2, 3)) * ratio).tril() @ u)
            state = torch.exp(last) * state + (torch.exp(last - b) * kc).transpose(2, 3) @ u
        else:
            qh, kh = qc * torch.exp(b), kc * torch.exp(-b)
            outs.append((qh @ kh.transpose(2, 3)).tril() @ vc + qh @ state)
            state = torch.exp(last).transpose(2, 3) * (state + kh.transpose(2, 3) @ vc)
    return torch.cat(outs, 2), state


def _exact_layer(case, q, k, v, decay, lq, lk, beta, h0):
    variant, (B, T, H) = case["variant"], q.shape[:3]
    gq, gk = torch.softmax(lq, -1).unsqueeze(-1), torch.softmax(lk, -1).unsqueeze(-1)
    q = gq * q
    if variant == "gdn":
        v = gk * v
    else:
        k = gk * k
    g = decay if variant == "gla" else (decay.view(1, 1, H, 1).expand(B, T, H, 1) if variant == "retnet" else decay.unsqueeze(-1))
    beta = beta.unsqueeze(-1) if variant == "gdn" else None
    cuts = _lengths(case) if case["kind"] == "packed" else [0, T]
    lens = [b - a for a, b in zip(cuts, cuts[1:])]
    parts = [x.transpose(1, 2).split(lens, 2) if x is not None else [None] * len(lens) for x in (q, k, v, g, beta)]
    outs, states = [], []
    for i in range(len(lens)):
        start = h0 if h0 is not None else q.new_zeros(B, H, case["dk"], case["dv"])
        o, st = _exact_sequence(variant, *(p[i] for p in parts), start)
        outs.append(o)
        states.append(st)
    return torch.cat(outs, 2).transpose(1, 2), torch.cat(states)


def _exact_feature_map(x, taps, normalize):
    B, T, H, d = x.shape
    padded = torch.nn.functional.pad(x.reshape(B, T, H * d), (0, 0, 3, 0))
    y = sum(taps[:, j] * padded[:, j:j + T] for j in range(4)).view(B, T, H, d)
    z = y * torch.sigmoid(y)
    return z / torch.sqrt((z * z).sum(-1, keepdim=True) + 1e-6) if normalize else z


def exact(case, seed):
    s = prepare(case, seed)
    kind, variant = case["kind"], case["variant"]
    x = {n: t.double() for n, t in s.items() if isinstance(t, torch.Tensor) and n not in ("ht", "ws")}
    del s
    if kind in ("decode", "prefill"):
        if x["q"].dim() == 3:                                # one token a call: no token axis
            t = {n: x[n].unsqueeze(1) for n in ("q", "k", "v", "lq", "lk") + (("beta",) if variant == "gdn" else ())}
            t["decay"] = x["decay"] if variant == "retnet" else x["decay"].unsqueeze(1)
        else:
            t = x
        with torch.no_grad():
            o, st = _exact_layer(case, t["q"], t["k"], t["v"], t["decay"], t["lq"], t["lk"], t.get("beta"),
                                 x.get("state", x.get("h0")))
        return dict(o=o, ht=st) if kind == "prefill" else dict(o=o.reshape(x["q"].shape[:-1] + (case["dv"],)), state=st)
    grads = {n: t.requires_grad_() for n, t in x.items() if n not in ("dO", "dy", "h0")}
    if kind != "layer":
        o, st = _exact_layer(case, x["q"], x["k"], x["v"], x["decay"], x["lq"], x["lk"], x.get("beta"), x.get("h0"))
        o.backward(x["dO"])
        return dict(o=o.detach(), ht=st.detach(), dq=grads["q"].grad, dk=grads["k"].grad, dv=grads["v"].grad,
                    dlog_decay=None if variant == "retnet" else grads["decay"].grad,
                    dbeta=grads["beta"].grad if variant == "gdn" else None,
                    dgq_logits=grads["lq"].grad, dgk_logits=grads["lk"].grad, dh0=None)
    q, k, v = x["x_q"], x["x_k"], x["x_v"]
    if variant == "gdn":
        q, k, v = (_exact_feature_map(x["x_" + n], x["taps_" + n], n != "v") for n in "qkv")
    lq, lk = (torch.einsum("bthc,ch->bth", t, x[w]) for t, w in ((q, "w_gq"), (k, "w_gk")))
    o, _ = _exact_layer(case, q, k, v, x["decay"], lq, lk, x.get("beta"), None)
    y = o.flatten(2) @ x["w_o"]
    y.backward(x["dy"])
    out = dict(y=y.detach(), dw_o=x["w_o"].grad, dw_gq=x["w_gq"].grad, dw_gk=x["w_gk"].grad,
               dlog_decay=None if variant == "retnet" else x["decay"].grad,
               dbeta=x["beta"].grad if variant == "gdn" else None)
    for n in "qkv":
        out["dx_" + n] = x["x_" + n].grad
        if variant == "gdn":
            out["dtaps_" + n] = x["taps_" + n].grad
    return out
