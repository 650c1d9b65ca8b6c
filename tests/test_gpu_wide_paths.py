"""Branches for the widest masks and the fullest windows: prefix masks of the
tuple kernel outside its lists, in shared memory and in global scratch, and
rank-indexed 2-hop windows whose mask words take several passes or do not fit
the staging memory. Counts are exact."""
from math import comb

import numpy as np
import pytest

import sbc_synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sbc():
    import torch

    assert torch.cuda.is_available()
    torch.cuda.init()
    import paper_2605_03603_gb300 as m

    return m


def dense(m, n, density, flip, seed):
    rng = np.random.default_rng(seed)
    u, v = np.divmod(np.arange(m * n, dtype=np.int64), n)
    keep = rng.random(m * n) < density
    s = (rng.choice([-1, 1], m)[u] * rng.choice([-1, 1], n)[v]).astype(np.int8)
    s[rng.random(m * n) < flip] *= -1
    return sbc_synth.from_edges(m, n, u[keep], v[keep], s[keep])


@pytest.mark.parametrize("m,n,p", [
    (260, 3200, 4),   # three partners: lists of more than 24,576 words, masks in shared memory,
    (40, 25000, 4),   # ... and in global scratch (two masks of 782 words)
    (16, 17000, 5),   # four partners, three masks of 532 words
    (14, 9000, 8),    # seven partners, six masks of 282 words
    # first rows by the CTA, in lists: 1 to 8 blocks of 32 entries, whose words the
    # warps share, and 9 and 10 blocks
    (40, 9000, 4),
    (300, 2500, 4),
    (24, 600, 5),
])
@pytest.mark.parametrize("density,flip", [(1.0, 0.0), (0.95, 0.02)])
def test_prefix_masks_outside_the_lists(sbc, m, n, p, density, flip):
    """Tuples of p with q = 2 on U against the other side, where a pair of anchors
    has one partner and its counters give the sum (no masks at all)."""
    g = dense(m, n, density, flip, seed=m + p)
    same_on_both_sides(sbc, g, p)


def same_on_both_sides(sbc, g, p):
    with sbc.graph_from_synth(g) as h:
        got, _, per = sbc.sbc_count_ex(h, p, 2, anchor_side=0, per_anchor=True, method="candidate")
        assert got == sum(per) == sbc.sbc_count_ex(h, p, 2, anchor_side=1)[0]
        assert got > 0


@pytest.mark.parametrize("m,n,p", [(60, 20000, 4), (60, 3001, 4), (45, 1999, 5), (30, 700, 6)])
@pytest.mark.parametrize("density,flip", [(0.5, 0.1), (0.3, 0.02)])
def test_projection_shared_by_warps(sbc, m, n, p, density, flip):
    """Rows of both parts, of unequal lengths: list words cut anywhere between the
    warps' ranges of mask words."""
    same_on_both_sides(sbc, dense(m, n, density, flip, seed=n), p)


@pytest.mark.parametrize("m,n,shards", [
    (24000, 40, 800),   # up to 23,999 rows and more in a window: set in global memory
    (900, 1100, 60),    # 35 words of 899 rows: two passes, positions in three batches each
])
@pytest.mark.parametrize("p,q", [(2, 2), (3, 3)])
def test_full_windows_equal_hash_tables(sbc, m, n, shards, p, q):
    """Every anchor takes the rank-indexed counters (one read per wedge for (2,2),
    where a hash window reads twice and buckets have an entry of their own in the
    statistics); with Algorithm 2's statistics the same anchors take the hash tables."""
    g = dense(m, n, 0.98, 0.02, seed=n)
    kw = dict(anchor_side=0, per_anchor=True, shard=0, shard_count=shards)
    with sbc.graph_from_synth(g) as h:
        got, st, per = sbc.sbc_count_ex(h, p, q, check=True, **kw)
        want, _, per_hash = sbc.sbc_count_ex(h, p, q, paper_tuples=True, **kw)
        _, pairs, _ = sbc.sbc_count_ex(h, 2, 2, **kw)
    assert got == want == sum(per) > 0
    assert per == per_hash
    n_anchors = (m + shards - 1) // shards
    assert st["twohop_anchors"] == [n_anchors, 0, 0, 0]
    assert pairs["twohop_reads"] == pairs["wedges"]


@pytest.mark.parametrize("m", [33, 290, 1000, 1025, 2050, 4001])
@pytest.mark.parametrize("p,q", [(4, 2), (6, 5)])
def test_column_walk_words(sbc, m, p, q):
    """Column masks of 1 to 126 words, cut anywhere within a block of words, leaves
    on both sides of the binomial table's end."""
    g = dense(m, 9, 1.0, 0.0, seed=m)
    with sbc.graph_from_synth(g) as h:
        got, _, per = sbc.sbc_count_ex(h, p, q, anchor_side=0, per_anchor=True, method="position")
    assert got == comb(m, p) * comb(9, q)
    assert sorted(per) == sorted(comb(r, p - 1) * comb(9, q) for r in range(m))


@pytest.mark.parametrize("m,n", [(130, 14), (420, 13), (700, 12)])
@pytest.mark.parametrize("p,q", [(4, 3), (5, 2)])
def test_column_walk_equals_rows(sbc, m, n, p, q):
    g = dense(m, n, 0.7, 0.15, seed=m)
    kw = dict(anchor_side=0, per_anchor=True, shard=0, shard_count=m // 8)
    with sbc.graph_from_synth(g) as h:
        walk, _, per = sbc.sbc_count_ex(h, p, q, method="position", **kw)
        rows, _, want = sbc.sbc_count_ex(h, p, q, method="candidate", **kw)
    assert walk == rows == sum(per) > 0
    assert per == want
