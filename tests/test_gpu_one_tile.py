"""Compaction of batches of one scan tile (2,048 rows), whose scan and gather
are one launch, and of the next size up, against the oracle: exact row lists,
counts, offsets and rows, with all, some and no rows kept and a capacity that
cuts them off."""

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


@pytest.mark.parametrize("rows", [(1,), (7, 1, 9), (2047,), (1024, 1024), (2000, 49), tuple([1] * 2048)])
@pytest.mark.parametrize("n_tensors", [1, 3, 8])
def test_compact_edges(rows, n_tensors):
    import paper_2605_29657_gb300 as occ

    rng = np.random.default_rng(sum(rows) + n_tensors)
    off = np.concatenate([[0], np.cumsum(rows)]).astype(np.int64)
    n, B = int(off[-1]), len(rows)
    lay = occ.BatchLayout(off, off, off[:-1].astype(np.int32), np.arange(B + 1, dtype=np.int32), np.arange(B + 1))
    # rows of 16 bytes, of a few, and of more than the eight 512-byte steps at once
    ts = [torch.randint(-30000, 30000, (n, (8, 24, 2056)[i % 3]), generator=torch.Generator().manual_seed(i),
                        dtype=torch.int16) for i in range(n_tensors)]
    for share, cap in ((1.0, n), (0.4, n), (0.4, max(1, n // 5)), (0.0, n), (1.0, 1)):
        keep = (rng.random(n) < share).astype(np.uint8)
        want, cnt, o, gathered = O.compact(keep.astype(bool), off, [t.numpy() for t in ts])
        ws = occ.alloc_workspace(lay, 1, 1)
        out = occ.occam_compact(lay, torch.from_numpy(keep).cuda(), [t.cuda() for t in ts], capacity_rows=cap, ws=ws)
        m = min(len(want), cap)
        assert occ.occam_get_status(ws) == (occ._lib.OCCAM_ERR_CAPACITY if len(want) > cap else 0)
        assert out["out_off"].tolist() == o.tolist() and out["count_out"].tolist() == cnt.tolist()
        assert out["out_index"][:m].tolist() == want[:m].tolist()
        for got, exact in zip(out["gathered"], gathered):
            assert (got[:m].cpu().numpy() == exact[:m]).all()
