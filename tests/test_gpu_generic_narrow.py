"""fp32 kernels for heads of at most 64 x 64 (two groups of threads, triangular products by 16 x 16 blocks): head widths, chunk sizes and last
chunks at the edges of the blocks, and the first shapes past them, against the fp64 oracle."""
import numpy as np
import pytest

from paper_2602_01744_b200.inputs import CONFIGS, make_inputs, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


# base: C0 Softmax-RetNet, C1 Softmax-GLA, C4 Softmax-GatedDeltaNet
@pytest.mark.parametrize("base,T,dk,dv,chunk,dtype", [
    ("C0", 1, 64, 64, 64, "fp32"), ("C0", 145, 64, 16, 64, "fp32"), ("C0", 161, 16, 64, 64, "fp32"), ("C0", 127, 48, 48, 64, "fp32"),
    ("C1", 63, 64, 64, 64, "fp32"), ("C1", 113, 64, 64, 64, "fp32"), ("C1", 79, 16, 16, 16, "fp32"), ("C1", 81, 32, 64, 32, "fp32"),
    ("C1", 96, 48, 32, 64, "bf16"), ("C4", 97, 64, 64, 64, "fp32"), ("C4", 49, 48, 64, 32, "fp32"),
    ("C1", 113, 80, 64, 64, "fp32"), ("C0", 113, 64, 80, 64, "fp32"),
    ("C0", 384, 32, 32, 16, "fp32"), ("C0", 385, 32, 32, 16, "fp32")])        # 144 and 150 chunks: on either side of one a SM
def test_step_matches_the_oracle(base, T, dk, dv, chunk, dtype):
    cfg = small(CONFIGS[base], B=2, T=T, H=3, d_k=dk, d_v=dv, chunk=chunk, dtype=dtype, seed=2300 + T, backward=True)
    x = make_inputs(cfg, with_dO=True, with_h0=True)
    xd = gu.to_dev(x)
    o, ht, g, *_ = gu.gpu_training_step(cfg, xd, h0=xd["h0"], dht=xd["dht"], want_dh0=True)
    oref, htref = gu.oracle_forward(cfg, x, h0=x["h0"])
    ref = gu.oracle_backward(cfg, x, h0=x["h0"], dht=x["dht"])
    pairs = {"o": (o, oref), "ht": (ht, htref)}
    pairs.update({n: (g[n], ref[r]) for n, r in gu.GRAD_NAMES.items() if g.get(n) is not None and np.linalg.norm(ref[r]) > 0})
    gu.assert_close({n: gu.rel_l2(a, r) for n, (a, r) in pairs.items()},
                    {n: gu.row_err(a, r) for n, (a, r) in pairs.items()}, cfg.dtype, cfg)
