"""The feature map's reverse pass in units of neighbouring tokens: sequences shorter than the taps and than a unit, more sequences than
thread groups, several and partly filled channel slabs - against the oracle."""
import pytest
import torch

from oracle import sla_oracle as orc
from paper_2602_01744_b200 import api
from paper_2602_01744_b200.inputs import CONFIGS, make_frontend_inputs, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,H,d,K", [(1, 1, 1, 16, 4), (1, 3, 5, 64, 4), (700, 5, 4, 64, 3), (2, 97, 32, 128, 4), (1, 2, 20, 64, 2), (3, 1200, 1, 32, 4)])
@pytest.mark.parametrize("normalize", [True, False])
def test_reverse_pass_at_the_edges_of_units(B, T, H, d, K, normalize):
    cfg = small(CONFIGS["C4"], B=B, T=T, H=H, d_k=d, d_v=d, seed=2400 + T)
    f = make_frontend_inputs(cfg, K, seed=2401)
    plan = api.sla_plan_create(cfg.variant, cfg.dtype, B, T, H, d, d, cfg.chunk)
    dx, dw = api.sla_shortconv_backward(plan, f["x_q"].cuda(), f["w_q"].cuda(), f["dout"].cuda(), normalize)
    torch.cuda.synchronize()
    dx_ref, dw_ref = orc.shortconv_backward(f["x_q"], f["w_q"], f["dout"], normalize)
    assert gu.rel_l2(dx, dx_ref) <= gu.TOL["bf16"] and gu.row_err(dx, dx_ref) <= gu.ROW_TOL["bf16"]
    assert gu.rel_l2(dw, dw_ref) <= gu.TOL["bf16"]


# groups of 32, 64, 96, 160 and 224 threads (four channels each), as many as a CTA holds, and the first shape of two slabs
@pytest.mark.parametrize("B,T,H,d,K", [(1, 5000, 1, 64, 4), (3, 1500, 4, 64, 4), (2, 900, 3, 128, 4), (1, 1200, 10, 64, 3), (40, 33, 7, 128, 4), (1, 700, 17, 64, 4)])
@pytest.mark.parametrize("normalize", [True, False])
def test_groups_as_wide_as_the_channels(B, T, H, d, K, normalize):
    test_reverse_pass_at_the_edges_of_units(B, T, H, d, K, normalize)
