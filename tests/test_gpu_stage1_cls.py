"""[CLS] Stage I of 72-dim heads at the edges of its tiles, against the oracle."""

from __future__ import annotations

import numpy as np
import pytest
import torch

from oracle import occam_oracle as O
from synth import tiny_batch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()
    assert torch.cuda.is_available()


@pytest.mark.parametrize("P", [(1, 2), (15, 16, 17), (700, 31, 1)])
def test_stage1_cls_72_dim_heads_edges(P):
    """[CLS] logits of 72-dim heads (a thread per row and head): segments that
    begin inside a 16-row tile, a last tile of few rows, one row in all. fp32
    sums of 72 products of N(0, 1) values are off by about 1e-7 of the largest
    partial sum (below 100), so the probabilities by 1e-5 at the very most."""
    import paper_2605_29657_gb300 as occ

    b = tiny_batch(B=len(P), segs=2, P=P, R=1, M=(3,) * len(P), H1=16, d1=72, H2=4, d2=128, hidden=64, seed=len(P),
                   beta1=2.0)
    m = b["meta"]
    layout = occ.BatchLayout.from_batch(b, "cuda")
    s1, ref1 = occ.occam_score_stage1(layout, occ.OCCAM_STAGE1_CLS, b["q_cls"].cuda(), b["K1"].cuda(),
                                      k_cls=b["k_cls"].cuda())
    w1, wr = O.stage1_cls(b["q_cls"], b["k_cls"], b["K1"], m["seg_off_host"], m["reg_idx_host"], m["reg_off_host"])
    np.testing.assert_allclose(s1.cpu().numpy(), w1, rtol=1e-5, atol=0)
    np.testing.assert_allclose(ref1.cpu().numpy(), wr, rtol=1e-5, atol=0)
