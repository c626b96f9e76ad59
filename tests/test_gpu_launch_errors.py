"""A call whose launch the CUDA runtime refuses answers SLA_ERR_CUDA, once: the next call, whose launches succeed, is not blamed for it."""
import pytest
import torch

from paper_2602_01744_b200 import api
from paper_2602_01744_b200.inputs import CONFIGS, make_inputs, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


def _refused(call):
    """Make `call` with the legacy default stream as its stream while a blocking stream is being captured: the runtime refuses every launch there
    (cudaErrorStreamCaptureImplicit) and nothing reaches the GPU."""
    from cuda.bindings import runtime as rt
    err, s = rt.cudaStreamCreate()
    assert int(err) == 0
    try:
        assert int(rt.cudaStreamBeginCapture(s, rt.cudaStreamCaptureMode.cudaStreamCaptureModeGlobal)[0]) == 0
        try:
            with pytest.raises(api.SLAError) as e:
                call()
        finally:
            rt.cudaStreamEndCapture(s)
    finally:
        rt.cudaStreamDestroy(s)
    assert e.value.status == 5                  # SLA_ERR_CUDA


# the chunk-parallel Gated-DeltaNet kernels, their one-CTA form, the segmented and the plain Softmax-GLA forward, the fp32 kernels
@pytest.mark.parametrize("base,B,T,H,dtype", [("C4", 1, 1100, 2, "bf16"), ("C4", 1, 100, 2, "bf16"), ("C1", 1, 1297, 2, "bf16"), ("C1", 1, 100, 2, "bf16"),
                                              ("C4", 1, 100, 2, "fp32")])
def test_a_refused_launch_is_reported_once(base, B, T, H, dtype):
    cfg = small(CONFIGS[base], B=B, T=T, H=H, dtype=dtype, seed=1800)
    x = gu.to_dev(make_inputs(cfg, with_dO=True))
    args = (x["q"], x["k"], x["v"], x["log_decay"], x["gq_logits"], x["gk_logits"])
    plan = api.sla_plan_create(cfg.variant, cfg.dtype, B, T, H, cfg.d_k, cfg.d_v)
    ws = plan.workspace(backward=True)
    o = torch.empty_like(x["v"])
    good = api.sla_forward(plan, *args, beta=x["beta"], o=torch.empty_like(o), workspace=ws)[0]
    grads = api.sla_backward(plan, *args, x["dO"], beta=x["beta"], workspace=ws)
    out = {n: None if t is None else torch.empty_like(t) for n, t in grads.items()}
    assert torch.cuda.current_stream().cuda_stream == 0         # the legacy default stream
    torch.cuda.synchronize()
    _refused(lambda: api.sla_forward(plan, *args, beta=x["beta"], o=o, workspace=ws))
    api.sla_forward(plan, *args, beta=x["beta"], o=o, workspace=ws)
    _refused(lambda: api.sla_backward(plan, *args, x["dO"], beta=x["beta"], workspace=ws, out=out))
    api.sla_backward(plan, *args, x["dO"], beta=x["beta"], workspace=ws, out=out)
    torch.cuda.synchronize()
    plan.poll()
    assert torch.equal(o, good)
    for n, t in grads.items():
        if t is not None:
            assert torch.equal(t, out[n]), n
