"""The count kernels at the sizes where a tile, a table or a dispatch rule
changes: direct 2-hop counters against the hash tables, the plan's row groups,
the tensor-core pair tiles and the tuple kernel's lists. Complete bipartite
graphs whose signs come from two labelings have C(m, p) C(n, q) balanced
bicliques; every other graph is compared per anchor with another strategy and
in total with the other anchor side. All counts are exact."""
from math import comb

import numpy as np
import pytest

import oracle
import sbc_synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sbc():
    import torch

    assert torch.cuda.is_available()
    torch.cuda.init()
    import paper_2605_03603_gb300 as m

    return m


def signed(n_u, n_v, u, v, flip, seed):
    rng = np.random.default_rng(seed)
    s = (rng.choice([-1, 1], n_u)[u] * rng.choice([-1, 1], n_v)[v]).astype(np.int8)
    s[rng.random(u.shape[0]) < flip] *= -1
    return sbc_synth.from_edges(n_u, n_v, u, v, s)


def block_graph(n_u, n_v, deg, step, flip, seed):
    """U vertex i has deg consecutive neighbours from i * step mod n_v on."""
    u = np.repeat(np.arange(n_u, dtype=np.int64), deg)
    v = (np.repeat(np.arange(n_u, dtype=np.int64) * step, deg) + np.tile(np.arange(deg), n_u)) % n_v
    o = np.lexsort((v, u))
    return signed(n_u, n_v, u[o], v[o], flip, seed)


@pytest.mark.parametrize("n_u,n_v,deg,step", [
    (300, 255, 255, 1),        # 8-bit counters, every count up to 255
    (300, 256, 256, 1),        # 16-bit counters
    (300, 512, 512, 1),        # positions in one batch,
    (300, 513, 513, 1),        # ... and in two
    (41500, 40, 3, 7),         # 8-bit counters, two windows of 40,960 ranks
    (21000, 20000, 256, 67),   # 16-bit counters, two windows of 20,480 ranks
])
@pytest.mark.parametrize("p,q", [(2, 2), (3, 3)])
def test_direct_counters_equal_hash_tables(sbc, n_u, n_v, deg, step, p, q):
    """The statistics of Algorithm 2 need the hash tables, so a count that asks
    for them is the same count on the general path."""
    g = block_graph(n_u, n_v, deg, step, 0.1, seed=n_v + p)
    with sbc.graph_from_synth(g) as h:
        got, st, per = sbc.sbc_count_ex(h, p, q, anchor_side=0, per_anchor=True, check=True)
        want, _, per_hash = sbc.sbc_count_ex(h, p, q, anchor_side=0, per_anchor=True,
                                             paper_tuples=True)
        plain = sbc.sbc_count_ex(h, p, q, anchor_side=0)[0]
    assert got == want == plain == sum(per)
    assert per == per_hash
    assert st["twohop_anchors"][0] > 0


def test_plan_row_groups(sbc):
    """Anchors of 1, 8, 9, 64, 65 (8 lanes to a warp per row), 1024 and 1025
    (warp to CTA) edges, per anchor against the oracle."""
    rng = np.random.default_rng(5)
    n_v, degs = 1100, [1, 8, 9, 63, 64, 65, 1023, 1024, 1025]
    u = np.concatenate([np.full(d, i * 4 + k, np.int64) for i, d in enumerate(degs) for k in range(4)])
    v = np.concatenate([np.sort(rng.choice(n_v, d, replace=False)) for d in degs for k in range(4)])
    g = signed(4 * len(degs), n_v, u, v, 0.1, seed=6)
    with sbc.graph_from_synth(g) as h:
        for p, q in ((2, 2), (3, 3)):
            got, _, per = sbc.sbc_count_ex(h, p, q, anchor_side=0, per_anchor=True)
            assert got == sum(per) == sbc.sbc_count_ex(h, p, q, anchor_side=1)[0]
            total, want = oracle.count(g, p, q, side=0, per_anchor=True)
            assert got == total
            assert per == [want[i] for i in range(g.n_u)]


@pytest.mark.parametrize("n,q", [
    (2, 2), (32, 2), (33, 2), (128, 2), (129, 2), (384, 2), (385, 2), (1023, 2), (1024, 2), (1500, 2),
    (102, 3), (103, 3), (203, 3), (204, 3), (33, 4), (34, 4), (55, 4), (56, 4), (129, 6),
])
def test_pair_tiles(sbc, n, q):
    """Every row count from 128 to 299 (tiles of 128 x 256 rows), one to twelve
    128-position steps (A rows beside up to three resident B blocks), rows on
    both sides of the epilogues' limits."""
    m = 300
    u, v = np.divmod(np.arange(m * n), n)
    g = signed(m, n, u, v, 0.0, seed=n)
    with sbc.graph_from_synth(g) as h:
        got, st, per = sbc.sbc_count_ex(h, 3, q, anchor_side=0, per_anchor=True, check=True,
                                        method="candidate")
    assert got == comb(m, 3) * comb(n, q)
    assert sorted(per) == sorted(comb(m - 1 - r, 2) * comb(n, q) for r in range(m))
    assert st["tc_anchors"] == m - 128


@pytest.mark.parametrize("n", [31, 33, 64, 65, 128, 129, 161])
@pytest.mark.parametrize("m,p,q", [(42, 4, 3), (42, 5, 2), (130, 4, 3), (30, 6, 4), (24, 7, 3), (20, 8, 2)])
def test_tuple_lists(sbc, m, n, p, q):
    """Lists around 40 and 128 rows, masks of one to six words, three to seven
    partners: row enumeration against the column walk and the other side."""
    rng = np.random.default_rng(1000 * m + n)
    u, v = np.divmod(np.arange(m * n), n)
    keep = rng.random(m * n) < 0.7
    g = signed(m, n, u[keep], v[keep], 0.15, seed=n)
    with sbc.graph_from_synth(g) as h:
        rows, _, per = sbc.sbc_count_ex(h, p, q, anchor_side=0, per_anchor=True, method="candidate")
        auto, _, per_auto = sbc.sbc_count_ex(h, p, q, anchor_side=0, per_anchor=True)
        assert rows == auto == sum(per)
        assert per == per_auto
        if q <= 3:
            assert rows == sbc.sbc_count_ex(h, p, q, anchor_side=1)[0]
        if n <= 65:
            assert rows == sbc.sbc_count_ex(h, p, q, anchor_side=0, method="position")[0]
    full = signed(m, n, u, v, 0.0, seed=n)
    with sbc.graph_from_synth(full) as h:
        assert sbc.sbc_count_ex(h, p, q, anchor_side=0)[0] == comb(m, p) * comb(n, q)
