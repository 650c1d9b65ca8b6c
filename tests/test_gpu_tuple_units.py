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


@pytest.mark.parametrize("split", [1, 4, 64])
@pytest.mark.parametrize("p,q", [(3, 3), (4, 4), (5, 5)])
@pytest.mark.parametrize("method", ["auto", "candidate", "position"])
def test_work_items_within_their_room(sbc, split, p, q, method):
    """One item per anchor and at most 2 x SMs x split_per_warp more, whichever
    path an anchor's plan names; the count is the same for every split."""
    import torch

    g = sbc_synth.plain_small()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with sbc.graph_from_synth(g) as h:
        want = sbc.sbc_count(h, p, q)
        for tc in (-1, 1):
            got, st, _ = sbc.sbc_count_ex(h, p, q, anchor_side=0, method=method,
                                          tune={"split_per_warp": split, "tc_min_words": tc})
            assert got == want
            assert st["work_items"] + st["tc_anchors"] <= g.n_u + 2 * sms * split
