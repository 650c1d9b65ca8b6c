"""The mask self-check (SBC_COUNT_CHECK) reads every word of every row: with it a
count popcounts the masks of all its rows once more than without, in every
2-hop tier. On a complete bipartite graph whose signs come from two labelings
an anchor with k later vertices has k rows of n positions."""
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


def labelled(m, n, seed):
    rng = np.random.default_rng(seed)
    u, v = np.divmod(np.arange(m * n, dtype=np.int64), n)
    s = (rng.choice([-1, 1], m)[u] * rng.choice([-1, 1], n)[v]).astype(np.int8)
    return sbc_synth.from_edges(m, n, u, v, s)


@pytest.mark.parametrize("m,n,shards,window", [
    (40, 9, 1, None),           # warp tier
    (300, 255, 1, None),        # rank-indexed counters of 8 bits,
    (300, 256, 1, None),        # ... of 16 bits,
    (300, 513, 1, None),        # ... with positions in two batches,
    (1100, 700, 97, None),      # ... masks in several ranges of positions, in batches,
    (24000, 40, 400, None),     # ... more rows in a window than its memory stages
    (300, 8, 1, "3583"),        # one hash window
    (300, 255, 16, "100"),      # hash windows from buckets
])
def test_every_row_is_checked(sbc, monkeypatch, m, n, shards, window):
    if window:
        monkeypatch.setenv("SBC_TWOHOP_WINDOW", window)
    g = labelled(m, n, seed=n)
    ranks = [r for r in range(0, m, shards)]
    rows = sum(m - 1 - r for r in ranks if m - 1 - r >= 2)
    with sbc.graph_from_synth(g) as h:
        kw = dict(anchor_side=0, shard=0, shard_count=shards)
        got, plain, _ = sbc.sbc_count_ex(h, 3, 3, **kw)
        again, st, _ = sbc.sbc_count_ex(h, 3, 3, check=True, **kw)
    assert got == again == sum(comb(m - 1 - r, 2) for r in ranks) * comb(n, 3)
    assert st["popc_words"] - plain["popc_words"] == rows * ((n + 31) // 32)
