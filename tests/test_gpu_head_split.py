"""Small batches whose text tiles have their heads split over several
clusters, against the oracle: tile counts at the edges of the rule (one tile;
as many as fit split; one more; more samples than the scratch serves), a
sample that 4-CTA clusters only just hold or do not, head counts whose groups
are not powers of two, ragged last tiles, and batches whose launches are left
out because they can have no items."""

from __future__ import annotations

import pytest
import torch

from synth import tiny_batch
from tests.gpu_helpers import check_prune, run_prune

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as g
    g.build()
    assert torch.cuda.is_available()


def _check(P, M, H2=32, H2kv=0, lam1=0.0, seed=0, **kw):
    b = tiny_batch(B=len(P), segs=1, P=tuple(P), R=3, M=tuple(M), H1=16, d1=64, H2=H2, d2=128, H2kv=H2kv, hidden=64,
                   seed=seed, beta1=2.0)
    gpu = run_prune(b, lam1, 1.1, **kw)
    assert gpu["status"] == 0
    check_prune(b, gpu, lam1, 1.1)
    return gpu


@pytest.mark.parametrize("M", [
    (128,),                        # one tile
    (129,),                        # two tiles of one sample: 8 groups of 4 heads on 4-CTA clusters
    (1, 128, 7),                   # three, one text row the fewest
    (200, 40, 300, 128),           # seven (every tile a resident 16-CTA cluster unsplit)
    (129, 257, 129, 1),            # eight
    tuple([130] * 9),              # 18: two groups, the most tiles that split
    tuple([130] * 9 + [3]),        # 19
    tuple([5] * 19),               # more samples than the scratch serves
])
def test_tile_counts(M):
    _check([40 + 9 * i for i in range(len(M))], M, seed=len(M))


@pytest.mark.parametrize("P", [(765, 50), (766, 50), (3069, 9)])
def test_sample_size_edges(P):
    """768 S1 keys just fit a 4-CTA cluster, 769 do not; 3,072 just fit 16 CTAs."""
    _check(P, (150, 20), seed=P[0])


@pytest.mark.parametrize("H2,H2kv", [(28, 4), (24, 8), (40, 8), (12, 12), (6, 2), (4, 1)])
def test_head_groups(H2, H2kv):
    """Groups of whole key heads, at least four query heads each; 4 and 6 heads do not split."""
    _check([90, 300, 33], (100, 129, 12), H2=H2, H2kv=H2kv, seed=H2)


def test_one_tile_that_may_need_the_two_pass_kernels():
    """One text tile, more rows than a 16-CTA cluster holds: the launches beside it stay."""
    _check([3300], (20,), seed=1)
    _check([3300], (20,), lam1=0.9, seed=1)


def test_split_equals_unsplit_route():
    b = tiny_batch(B=3, segs=2, P=(60, 200, 90), R=2, M=(140, 30, 128), H1=16, d1=64, H2=32, d2=128, hidden=64, seed=5,
                   beta1=2.0)
    a, z = run_prune(b, 0.2, 1.0), run_prune(b, 0.2, 1.0, path="narrow")
    # fp32 sums of 32 heads' probabilities in another grouping
    torch.testing.assert_close(torch.from_numpy(a["s2"]), torch.from_numpy(z["s2"]), rtol=4e-6, atol=1e-9)
    torch.testing.assert_close(torch.from_numpy(a["ref2"]), torch.from_numpy(z["ref2"]), rtol=4e-6, atol=1e-9)


@pytest.mark.parametrize("P,M", [
    ((900, 60, 400), (100, 130, 20)),                  # one sample on 8-CTA clusters beside two on 4
    ((1533, 1000), (129, 250)),                        # all on 8-CTA clusters; 1,536 keys just fit
    ((1534, 100), (20, 140)),                          # one that needs 16
    ((800,) + (90,) * 7, (64,) * 8),
])
def test_split_with_larger_samples(P, M):
    _check(P, M, seed=len(P) + P[0])


@pytest.mark.parametrize("P,M,H2", [
    ((576,), (32,), 32),                     # one tile, all rows fit 4-CTA clusters: that launch alone
    ((40, 300, 700), (128, 5, 64), 32),
    ((20, 30, 40, 50), (2, 130, 257, 4), 24),
    ((60,), (20,), 6),                       # heads that do not split
])
def test_four_cta_launch_alone(P, M, H2):
    _check(P, M, H2=H2, seed=sum(P))
    _check(P, M, H2=H2, lam1=0.6, seed=sum(P))


def test_as_many_segments_as_samples_with_one_sample_empty():
    """Two samples of two segments between two without a row: their S1 lists
    still follow the order of their segments."""
    P, M = (60, 200), (40, 30)
    b = tiny_batch(B=2, segs=2, P=P, R=2, M=M, H1=16, d1=64, H2=32, d2=128, hidden=64, seed=3, beta1=2.0)
    want = run_prune(b, 0.2, 1.0)
    m = dict(b["meta"])
    r = m["row_off_host"]
    # the last text token of each sample becomes a rowless sample's
    m["row_off_host"] = torch.tensor([0, r[1], r[1], r[2], r[2]]).numpy()
    m["text_off_host"] = torch.tensor([0, 39, 40, 69, 70]).numpy()
    got = run_prune(dict(b, meta=m), 0.2, 1.0)
    assert got["status"] == 0 == want["status"]
    for k in ("s1", "ref1", "keep1"):
        assert (got[k] == want[k]).all(), k
    assert got["n1_vis"][0::2].tolist() == want["n1_vis"].tolist()
    # the same samples with that text alone, each a batch of its own
    assert got["count_out"][1::2].tolist() == [0, 0]
    o = got["out_off"]
    assert (o[1::2] == o[2::2]).all() and o[4] == got["count_out"].sum()
    keep2 = got["keep2"].nonzero()[0]
    assert got["out_index"][:o[4]].tolist() == keep2.tolist()
    one = dict(b)
    m1 = dict(b["meta"])
    keep = [i for i in range(70) if i not in (39, 69)]
    one["Q_text"], one["K_text"] = b["Q_text"][keep], b["K_text"][keep]
    m1["text_off_host"] = torch.tensor([0, 39, 68]).numpy()
    one["meta"] = m1
    z = run_prune(one, 0.2, 1.0)
    # fp32 sums of 32 heads' probabilities in another grouping
    torch.testing.assert_close(torch.from_numpy(got["s2"]), torch.from_numpy(z["s2"]), rtol=4e-6, atol=1e-9)
