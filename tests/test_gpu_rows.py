"""The row-wise entry points (selection rules, register construction, lambda2
calibration) at the sizes where their kernels change path: units of one row,
register bits at the end of a word, more rows than a CTA takes at a time,
samples staged in shared memory and above, register bits in several windows,
rows of one cluster and above. Everything is compared exactly with the oracle
or with plain NumPy on the same fp32 values."""

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


def _layout(seg_rows, segs_per_sample, regs, seed):
    """Segments of the given row counts with `regs` registers each at random rows."""
    import paper_2605_29657_gb300 as occ

    rng = np.random.default_rng(seed)
    seg_off = np.concatenate([[0], np.cumsum(seg_rows)]).astype(np.int64)
    row_off = np.concatenate([[0], np.cumsum([sum(seg_rows[i:i + n]) for i, n in zip(
        np.cumsum([0] + segs_per_sample[:-1]), segs_per_sample)])]).astype(np.int64)
    reg, off = [], [0]
    for a, z in zip(seg_off[:-1], seg_off[1:]):
        k = min(regs, int(z - a))
        reg += sorted(rng.choice(np.arange(a, z), size=k, replace=False).tolist())
        off.append(len(reg))
    text = np.arange(len(row_off), dtype=np.int64)
    lay = occ.BatchLayout(row_off, seg_off, np.asarray(reg, np.int32), np.asarray(off, np.int32), text, device="cuda")
    is_reg = np.zeros(int(seg_off[-1]), bool)
    is_reg[reg] = True
    return lay, seg_off, row_off, is_reg, rng


# (segment rows, segments per sample, registers per segment)
SHAPES = [
    ([1, 31, 32, 33, 2], [1, 3, 1], 1),
    ([2047, 2048, 2049, 5000], [2, 2], 3),     # rows a threshold CTA takes at a time
    ([40960], [1], 4),                          # the largest staged sample of the budget rule
    ([40961, 7], [1, 1], 4),                    # above it
    ([65536, 65537, 100], [1, 1, 1], 5),        # register bits in one window, and above
]


@pytest.mark.parametrize("shape", range(len(SHAPES)))
@pytest.mark.parametrize("prev", [False, True])
def test_rules_at_unit_edges(shape, prev):
    import paper_2605_29657_gb300 as occ

    lay, seg_off, row_off, is_reg, rng = _layout(*SHAPES[shape], seed=100 + shape)
    n = int(row_off[-1])
    s = rng.integers(0, 200, n).astype(np.float32) / 16  # ties
    s[rng.random(n) < 0.02] = 0
    pk = (rng.random(n) < 0.6).astype(np.uint8) if prev else None
    cand = ~is_reg & (pk.astype(bool) if prev else True)
    ts, tp = torch.from_numpy(s).cuda(), torch.from_numpy(pk).cuda() if prev else None
    for scope, off in ((occ.OCCAM_REF_SEGMENT, seg_off), (occ.OCCAM_REF_SAMPLE, row_off)):
        want = O.mean_reference(s, off, cand).astype(np.float32)
        ref = occ.occam_mean_reference(lay, ts, scope, prev_keep=tp)
        # sums of multiples of 1/16 are exact in fp64 in any order
        assert (ref.cpu().numpy() == want).all()
        unit = np.repeat(np.arange(len(off) - 1), np.diff(off))
        for kr in (True, False):
            keep, cnt = occ.occam_threshold(lay, ts, ref, scope, 1.25, prev_keep=tp, keep_registers=kr)
            k = cand & (s >= np.float32(1.25) * want[unit])
            assert (keep.cpu().numpy().astype(bool) == (k | (is_reg & kr))).all()
            assert cnt.cpu().numpy().tolist() == np.add.reduceat(k, row_off[:-1]).tolist()
    nc = np.add.reduceat(cand, row_off[:-1])
    for budget in (np.zeros_like(nc), nc // 3 + 1, nc - 1, nc, nc + 5, -nc):
        want, cnt = O.budget_keep(s, row_off, cand, budget, is_reg, True)
        keep, got = occ.occam_budget_keep(lay, ts, torch.from_numpy(budget.astype(np.int32)).cuda(), prev_keep=tp)
        assert (keep.cpu().numpy().astype(bool) == want).all()
        assert got.cpu().numpy().tolist() == cnt.tolist()


@pytest.mark.parametrize("n_k", [1, 10, 255, 256, 257])
def test_construct_registers_channel_groups(n_k):
    """Up to 256 channels go through the CTA at once; 257 take a second group."""
    import paper_2605_29657_gb300 as occ

    lay, seg_off, _, _, rng = _layout([3, 300, 4100], [2, 1], 2, seed=n_k)
    h = torch.randn(int(seg_off[-1]), 300, generator=torch.Generator().manual_seed(n_k)).to(torch.bfloat16)
    k = rng.permutation(300)[:n_k].astype(np.int32)
    want = O.construct_registers(h.float().numpy(), seg_off, lay.host["reg_idx"], lay.host["reg_off"], k)
    got = occ.occam_construct_registers(lay, h.cuda(), torch.from_numpy(k).cuda())
    assert (got.float().cpu().numpy() == want).all()


def test_construct_registers_several_windows():
    """A segment of more rows than the register bits hold (two windows), and one without visual rows."""
    import paper_2605_29657_gb300 as occ

    lay, seg_off, _, _, _ = _layout([65536 + 70, 2], [1, 1], 2, seed=3)
    h = torch.randn(int(seg_off[-1]), 12, generator=torch.Generator().manual_seed(1)).to(torch.bfloat16)
    k = np.asarray([11, 0, 5], np.int32)
    want = O.construct_registers(h.float().numpy(), seg_off, lay.host["reg_idx"], lay.host["reg_off"], k)
    got = occ.occam_construct_registers(lay, h.cuda(), torch.from_numpy(k).cuda())
    assert (got.float().cpu().numpy() == want).all()


@pytest.mark.parametrize("seg_rows,segs", [
    ([5], [1]),                                  # fewer rows than CTAs
    ([17, 1, 300], [1, 2]),
    ([3] * 1200, [2] * 600),                     # more samples than are staged
    ([100000, 227680], [1, 1]),
    ([458752], [1]),                             # the most rows of the one-cluster kernel
    ([458753], [1]),                             # the grid-wide kernels
])
def test_calibrate_lambda2_row_ranges(seg_rows, segs):
    import paper_2605_29657_gb300 as occ

    lay, _, row_off, is_reg, rng = _layout(seg_rows, segs, 1, seed=len(seg_rows))
    n, B = int(row_off[-1]), len(segs)
    for spread, tiny in ((1.0, False), (1e-4, False), (1.0, True)):
        # wide, nearly tied (many quotients within the window), and products too small for the margin shortcut
        s2 = np.exp(spread * rng.standard_normal(n)).astype(np.float32)
        ref2 = np.exp(0.2 * rng.standard_normal(B)).astype(np.float32)
        if tiny:
            s2, ref2 = s2 * np.float32(1e-33), ref2 * np.float32(1e-16)
        ref2[rng.random(B) < 0.1] = 0
        keep1 = (rng.random(n) < 0.4).astype(np.uint8)
        args = [torch.from_numpy(x).cuda() for x in (s2, ref2, keep1)]
        nc = int((keep1.astype(bool) & ~is_reg & (ref2[np.repeat(np.arange(B), np.diff(row_off))] > 0)).sum())
        for K in sorted({0, 1, nc // 7, nc - 1, nc, nc + 1}):
            want, cnt = O.lambda2_for_budget(s2, ref2, keep1, is_reg, row_off, K)
            lam, got = occ.occam_calibrate_lambda2(lay, *args, K)
            assert int(got[0]) == cnt == nc
            assert np.float32(lam[0].item()) == want, (K, spread, tiny)


@pytest.mark.parametrize("rows", [[2048, 5], [2049, 1, 255, 257, 300], [16385, 2304, 1]])
def test_mean_reference_at_the_split(rows):
    """Units summed by one CTA (2,048 rows at most) and by eight."""
    import paper_2605_29657_gb300 as occ

    lay, seg_off, _, is_reg, rng = _layout(rows, [1] * len(rows), 1, seed=len(rows))
    n = int(seg_off[-1])
    s = rng.integers(0, 200, n).astype(np.float32) / 16
    pk = (rng.random(n) < 0.5).astype(np.uint8)
    for scope in (occ.OCCAM_REF_SEGMENT, occ.OCCAM_REF_SAMPLE):
        ref = occ.occam_mean_reference(lay, torch.from_numpy(s).cuda(), scope, prev_keep=torch.from_numpy(pk).cuda())
        # sums of multiples of 1/16 are exact in fp64 in any order
        assert (ref.cpu().numpy() == O.mean_reference(s, seg_off, ~is_reg & pk.astype(bool)).astype(np.float32)).all()
