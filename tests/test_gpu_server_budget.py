"""A server admits a job by an estimate of its device bytes: it covers what the
count of a graph of one-word masks takes at its peak, whose operands on the tensor
cores are 32 times the size of the masks."""
import ctypes
import threading
from math import comb

import numpy as np
import pytest

import sbc_synth

pytestmark = pytest.mark.gpu

ALLOC_FN = ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p, ctypes.c_void_p)
FREE_FN = ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p, ctypes.c_void_p)


@pytest.fixture(scope="module")
def sbc():
    import torch

    assert torch.cuda.is_available()
    torch.cuda.init()
    import paper_2605_03603_gb300 as m

    f = m.lib.sbc_set_allocator
    f.restype = ctypes.c_int
    f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]
    return m


@pytest.mark.parametrize("p,q", [(3, 4), (4, 3)])
def test_estimate_covers_the_peak(sbc, p, q):
    """100 blocks K_{200,30} with signs from two labelings, tuples of three on the
    side of 200: 72 anchors of each block have 128 rows and more."""
    import torch

    rng = np.random.default_rng(3)
    m, n, copies = (200, 30, 100) if p == 3 else (30, 200, 100)
    u, v = np.divmod(np.arange(m * n, dtype=np.int64), n)
    u = np.concatenate([u + c * m for c in range(copies)])
    v = np.concatenate([v + c * n for c in range(copies)])
    s = (rng.choice([-1, 1], copies * m)[u] * rng.choice([-1, 1], copies * n)[v]).astype(np.int8)
    g = sbc_synth.from_edges(copies * m, copies * n, u, v, s)
    live, now, peak, lock = {}, [0], [0], threading.Lock()

    def alloc(nbytes, stream, ctx):
        x = torch.cuda.caching_allocator_alloc(max(int(nbytes), 1))
        with lock:
            live[x] = int(nbytes)
            now[0] += int(nbytes)
            peak[0] = max(peak[0], now[0])
        return x

    def free(ptr, nbytes, stream, ctx):
        torch.cuda.synchronize()
        with lock:
            now[0] -= live.pop(int(ptr))
        torch.cuda.caching_allocator_delete(int(ptr))

    a, f = ALLOC_FN(alloc), FREE_FN(free)
    assert sbc.lib.sbc_set_allocator(ctypes.cast(a, ctypes.c_void_p), ctypes.cast(f, ctypes.c_void_p), None) == 0
    try:
        with sbc.graph_from_synth(g) as h:
            for side in (0, 1):
                sbc.sbc_count_ex(h, 2, 2, anchor_side=side)  # both sides resident
            with sbc.Server(lanes=1) as srv:
                gid = srv.add_graph(h)
                resident = peak[0] = now[0]
                got, _ = srv.wait(srv.submit(gid, p, q))
                taken = peak[0] - resident
                assert got == copies * comb(200, 3) * comb(30, 4)
                assert srv.stats()["peak_admitted_bytes"] >= taken > 200 << 20
    finally:
        assert sbc.lib.sbc_set_allocator(None, None, None) == 0
