"""The tuple kernel's work units: first rows deferred to the whole CTA in
several rounds. Counts are exact; complete bipartite graphs whose signs come
from two labelings have closed forms."""
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


def labelled_blocks(copies, m, n, seed):
    """`copies` disjoint K_{m,n} with signs from two labelings (every butterfly balanced)."""
    rng = np.random.default_rng(seed)
    u, v = np.divmod(np.arange(m * n, dtype=np.int64), n)
    u = np.concatenate([u + c * m for c in range(copies)])
    v = np.concatenate([v + c * n for c in range(copies)])
    s = (rng.choice([-1, 1], copies * m)[u] * rng.choice([-1, 1], copies * n)[v]).astype(np.int8)
    return sbc_synth.from_edges(copies * m, copies * n, u, v, s)


@pytest.mark.parametrize("m", [45, 240, 290])
def test_deferred_rows(sbc, m):
    """Lists of 40 rows and more go to the CTA: up to 250 first rows of one work
    item, more than the 240 after which a round ends. Six blocks, so that no
    anchor is split among items."""
    g = labelled_blocks(6, m, 8, seed=m)
    with sbc.graph_from_synth(g) as h:
        got, _, per = sbc.sbc_count_ex(h, 5, 2, anchor_side=0, per_anchor=True, method="candidate",
                                       tune={"split_per_warp": 1})
    assert got == 6 * comb(m, 5) * comb(8, 2)
    assert sorted(per) == sorted(comb(r, 4) * comb(8, 2) for r in range(m) for _ in range(6))
