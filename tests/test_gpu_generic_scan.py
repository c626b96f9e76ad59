"""GPU parity of the fp32 kernels' state passes (per-chunk products and the fold along the sequence for Softmax-RetNet and
-GLA, the chunk walk for Softmax-GDN) at the edges of their tiles: key widths below, between and at the 64-row blocks, value
widths that fill no 32-column block, ragged last chunks, more chunks than the fold reads ahead, every chunk size."""
import pytest
import torch

from paper_2602_01744_b200 import api
from paper_2602_01744_b200.inputs import CONFIGS, make_inputs, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base", ["C0", "C1", "C4"])
@pytest.mark.parametrize("B,T,H,dk,dv,chunk", [(1, 1, 1, 16, 16, 64), (2, 65, 3, 80, 48, 64), (1, 577, 2, 96, 112, 64),
                                               (1, 150, 2, 128, 128, 16), (2, 95, 2, 64, 64, 32)])
def test_state_passes_at_tile_edges(base, B, T, H, dk, dv, chunk):
    cfg = small(CONFIGS[base], B=B, T=T, H=H, d_k=dk, d_v=dv, chunk=chunk, dtype="fp32", seed=1700 + T, backward=True)
    assert max(gu.check_forward(small(cfg, backward=False), with_h0=True, flags=api.SLA_FLAG_FORCE_GENERIC).values()) <= 1e-4
    assert max(gu.check_backward(cfg, with_h0=True, flags=api.SLA_FLAG_FORCE_GENERIC).values()) <= 1e-4


# fp32 kernels with one chunk and several, the tensor-core kernels in one piece, in segments and (Softmax-GDN) chunk-parallel
@pytest.mark.parametrize("base,T,d,dtype", [("C0", 40, 64, "fp32"), ("C0", 300, 128, "fp32"), ("C1", 300, 48, "fp32"), ("C4", 300, 64, "fp32"),
                                            ("C1", 300, 128, "bf16"), ("C1", 2048, 128, "bf16"), ("C4", 300, 128, "bf16"), ("C4", 1100, 128, "bf16")])
def test_state_gradients_may_be_updated_in_place(base, T, d, dtype):
    """dh0 in the buffer that brought dht.  The fp32 kernels then add the first chunk's share in a step of its own: two more roundings, of values
    of the size of the largest entries, 2^-24 each."""
    cfg = small(CONFIGS[base], B=2, T=T, H=3, d_k=d, d_v=d, dtype=dtype, seed=1790 + T, backward=True)
    x = gu.to_dev(make_inputs(cfg, with_dO=True, with_h0=True))
    args = (x["q"], x["k"], x["v"], x["log_decay"], x["gq_logits"], x["gk_logits"], x["dO"])
    plan = api.sla_plan_create(cfg.variant, cfg.dtype, cfg.B, cfg.T, cfg.H, d, d)
    apart = api.sla_backward(plan, *args, beta=x["beta"], h0=x["h0"], dht=x["dht"], want_dh0=True)
    inplace = {n: None if t is None else torch.empty_like(t) for n, t in apart.items()}
    inplace["dh0"] = x["dht"].clone()
    api.sla_backward(plan, *args, beta=x["beta"], h0=x["h0"], dht=inplace["dh0"], out=inplace)
    torch.cuda.synchronize()
    plan.poll()
    for n, t in apart.items():
        if t is not None and n != "dh0":
            assert torch.equal(t, inplace[n]), n
    err = float((apart["dh0"].double() - inplace["dh0"].double()).abs().max())
    assert err <= 2.0 ** -22 * float(apart["dh0"].abs().max()), err
