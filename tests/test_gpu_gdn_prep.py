"""The chunk-parallel Softmax-GatedDeltaNet preparation fetches a worker's next chunk a chunk ahead: head counts of both gate forms (16-byte
blocks of logits; a row a thread), several chunks a worker, last chunks of one token and of 63, against the fp64 oracle."""
import numpy as np
import pytest

from paper_2602_01744_b200.inputs import CONFIGS, make_inputs, small
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


# chunks = B x H x ceil(T / 64); 444 workers on 148 SMs: 1 .. 3 chunks each, neighbours of other sequences and heads
@pytest.mark.parametrize("B,T,H", [(9, 1025, 4), (3, 1151, 8), (2, 1089, 16), (1, 1087, 32), (13, 1025, 5), (5, 1151, 12)])
def test_step_matches_the_oracle(B, T, H):
    cfg = small(CONFIGS["C4"], B=B, T=T, H=H, d_k=64, d_v=64, seed=1900 + T + H)
    x = make_inputs(cfg, with_dO=True)
    o, ht, g, plan, ws, lf, lb = gu.gpu_training_step(cfg, gu.to_dev(x))
    assert (lf, lb) == (1, 2)
    oref, htref = gu.oracle_forward(cfg, x)
    ref = gu.oracle_backward(cfg, x)
    pairs = {"o": (o, oref), "ht": (ht, htref)}
    pairs.update({n: (g[n], ref[r]) for n, r in gu.GRAD_NAMES.items() if g.get(n) is not None and np.linalg.norm(ref[r]) > 0})
    gu.assert_close({n: gu.rel_l2(a, r) for n, (a, r) in pairs.items()},
                    {n: gu.row_err(a, r) for n, (a, r) in pairs.items()}, cfg.dtype, cfg)
