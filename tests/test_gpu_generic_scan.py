"""GPU parity of the fp32 kernels' state passes (per-chunk products and the fold along the sequence for Softmax-RetNet and
-GLA, the chunk walk for Softmax-GDN) at the edges of their tiles: key widths below, between and at the 64-row blocks, value
widths that fill no 32-column block, ragged last chunks, more chunks than the fold reads ahead, every chunk size."""
import pytest

from paper_2602_01744_b200 import api
from paper_2602_01744_b200.inputs import CONFIGS, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base", ["C0", "C1", "C4"])
@pytest.mark.parametrize("B,T,H,dk,dv,chunk", [(1, 1, 1, 16, 16, 64), (2, 65, 3, 80, 48, 64), (1, 577, 2, 96, 112, 64),
                                               (1, 150, 2, 128, 128, 16), (2, 95, 2, 64, 64, 32)])
def test_state_passes_at_tile_edges(base, B, T, H, dk, dv, chunk):
    cfg = small(CONFIGS[base], B=B, T=T, H=H, d_k=dk, d_v=dv, chunk=chunk, dtype="fp32", seed=1700 + T, backward=True)
    assert max(gu.check_forward(small(cfg, backward=False), with_h0=True, flags=api.SLA_FLAG_FORCE_GENERIC).values()) <= 1e-4
    assert max(gu.check_backward(cfg, with_h0=True, flags=api.SLA_FLAG_FORCE_GENERIC).values()) <= 1e-4
