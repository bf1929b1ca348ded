"""Mutual Stage I on CTA pairs (batches of long segments on average) and on
single CTAs (short ones), at the edges of their tiles (256 rows an item, 128 a
CTA, blocks of 256 keys taken in turn by two groups of softmax warps), with
head counts that leave a ragged head group, and with logits that overflow the
pairs' first pass's running sums (items worked through a second time)."""

from __future__ import annotations

import numpy as np
import pytest
import torch

from oracle import occam_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()
    assert torch.cuda.is_available()


def _check(rows, H, d, seed, scale=None, rtol=4e-6, plain=False):
    import paper_2605_29657_gb300 as occ

    g = torch.Generator().manual_seed(seed)
    off = np.concatenate([[0], np.cumsum(rows)]).astype(np.int64)
    S = len(rows)
    Q = torch.randn(int(off[-1]), H, d, generator=g).to(torch.bfloat16)
    K = torch.randn(int(off[-1]), H, d, generator=g).to(torch.bfloat16)
    if scale is not None:
        K = (K.float() * scale(off)[:, None, None]).to(torch.bfloat16)
    reg = (off[1:] - 1).astype(np.int32)
    lay = occ.BatchLayout(off, off, reg, np.arange(S + 1, dtype=np.int32), np.arange(S + 1, dtype=np.int64))
    ws = occ.alloc_workspace(lay, H, 1)
    s1, ref1 = occ.occam_score_stage1(lay, occ.OCCAM_STAGE1_MUTUAL, Q.cuda(), K.cuda(), ws=ws)
    assert occ.occam_get_status(ws) == 0
    if plain:
        # the oracle's sums, in fp64 on the device (the batch is too large for it)
        want = torch.empty(int(off[-1]), dtype=torch.float64)
        for a, z in zip(off[:-1], off[1:]):
            q, k = Q[a:z].cuda().double(), K[a:z].cuda().double()
            want[a:z] = sum(torch.softmax(q[:, h] @ k[:, h].T / d ** 0.5, 1).sum(0) for h in range(H)).cpu() / (H * (z - a))
        want = want.numpy()
        wref = want[reg]
    else:
        want, wref = O.stage1_mutual(Q, K, off, reg, np.arange(S + 1))
    # fp32 logits of |l| <= about 50 in log2 units are off by up to 2^-24 * 50
    # = 3e-6, as are the probabilities relatively; the sums average below that
    np.testing.assert_allclose(s1.cpu().numpy(), want, rtol=rtol, atol=1e-9)
    np.testing.assert_allclose(ref1.cpu().numpy(), wref, rtol=rtol, atol=1e-9)


@pytest.mark.parametrize("d", [64, 72, 80])
@pytest.mark.parametrize("H", [1, 3, 16])
def test_tile_edges(d, H):
    edges = [2, 127, 128, 129, 255, 256, 257, 384, 385, 511, 513, 769]
    _check(edges, H, d, seed=d + H)
    # two long segments bring the mean past the line to the pairs
    _check([5900] + edges + [6000], H, d, seed=d + H, plain=True)


@pytest.mark.parametrize("d,H", [(72, 10), (64, 6)])
def test_head_groups_of_a_larger_batch(d, H):
    """Enough tiles for items of four heads, with a ragged last group."""
    _check([1500, 1100, 1300, 900] * (20 if H > 8 else 30), H, d, seed=7, plain=True)


@pytest.mark.parametrize("d", [64, 72, 80])
def test_overflowing_sums_are_redone(d):
    """Keys past a segment's first 33 up to 256 times larger: their logits lie
    hundreds of log2 units above the first piece's, so the first pass's sums
    overflow for most rows of the scaled segments, beside one untouched. The
    probabilities are then those of logits of up to some 2,000 units, off by
    2^-24 of that."""
    def scale(off):
        f = np.ones(int(off[-1]), np.float32)
        f[off[0] + 33:off[1]] = 256
        f[off[2] + 300:off[3]] = 128
        return torch.from_numpy(f)

    _check([1500, 900, 1300], 4, d, seed=d, scale=scale, rtol=1e-3)
    _check([600, 300, 700], 4, d, seed=d, scale=scale, rtol=1e-3)  # (single CTAs)
