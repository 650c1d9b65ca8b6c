"""Blocks that outlive the stream they were allocated on: a graph's orientation
built by a server's lane, a batch made on a stream of the caller's. Their frees
must not name that stream once it may be gone."""
import ctypes

import pytest

import oracle
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


class RecordingAllocator:
    """Device memory from torch through the allocator hook; `frees` lists the
    streams the library freed on (0: the default stream). The block numbered
    `fail_at` (1-based, counted in `calls`) is refused."""

    def __init__(self, sbc, fail_at=0):
        import torch

        self.torch, self.sbc = torch, sbc
        self.live, self.frees = {}, []
        self.fail_at, self.calls = fail_at, 0
        self._a, self._f = ALLOC_FN(self._alloc), FREE_FN(self._free)

    def _alloc(self, nbytes, stream, ctx):
        self.calls += 1
        if self.calls == self.fail_at:
            return None
        p = self.torch.cuda.caching_allocator_alloc(max(int(nbytes), 1))
        self.live[p] = stream or 0
        return p

    def _free(self, ptr, nbytes, stream, ctx):
        self.torch.cuda.synchronize()
        self.frees.append(stream or 0)
        self.live.pop(int(ptr))
        self.torch.cuda.caching_allocator_delete(int(ptr))

    def __enter__(self):
        assert self.sbc.lib.sbc_set_allocator(ctypes.cast(self._a, ctypes.c_void_p),
                                              ctypes.cast(self._f, ctypes.c_void_p), None) == 0
        return self

    def __exit__(self, *exc):
        assert self.sbc.lib.sbc_set_allocator(None, None, None) == 0


def two_sided():
    """A graph counted on U for (3,4) and on V for (4,3)."""
    return sbc_synth.chung_lu_signed(41, 900, 800, 9000, 2.2, 2.2, 0.2)


def test_graph_outlives_the_lane_that_built_a_side(sbc):
    g = two_sided()
    with RecordingAllocator(sbc) as a:
        h = sbc.graph_from_synth(g)
        with sbc.Server(lanes=2) as srv:
            gid = srv.add_graph(h)
            got = [srv.wait(srv.submit(gid, p, q))[0] for p, q in ((3, 4), (4, 3))]
        assert any(a.live.values())  # a side is held in blocks of a lane's stream
        a.frees.clear()
        h.close()
        assert a.frees and not any(a.frees)
        assert not a.live
    assert got == [oracle.count(g, 3, 4, side=0), oracle.count(g, 4, 3, side=0)]


def test_batch_outlives_the_stream_it_was_made_on(sbc, monkeypatch):
    """Several anchor groups: every run plans again, on its own stream."""
    import torch

    g = two_sided()
    want = oracle.count(g, 3, 3, side=0)
    made, ran = torch.cuda.Stream(), torch.cuda.Stream()
    monkeypatch.setenv("SBC_POOL_BUDGET_KB", "4")
    with RecordingAllocator(sbc) as a:
        h = sbc.graph_from_synth(g)
        b = sbc.Batch([h, h], 3, 3, stream=made)
        a.frees.clear()
        assert b.run(stream=ran) == [want, want]
        assert a.frees and made.cuda_stream not in a.frees
        a.frees.clear()
        b.close()
        h.close()
        assert a.frees and not any(a.frees)
        assert not a.live


def test_closing_order_is_free(sbc):
    """Server first, then the graphs it had oriented, then counts again, without a hook."""
    g = two_sided()
    want = [oracle.count(g, 3, 4, side=0), oracle.count(g, 4, 3, side=0)]
    for _ in range(3):
        h = sbc.graph_from_synth(g)
        srv = sbc.Server(lanes=2)
        gid = srv.add_graph(h)
        got = [srv.wait(srv.submit(gid, p, q))[0] for p, q in ((3, 4), (4, 3))]
        srv.close()
        again = [sbc.sbc_count(h, 3, 4), sbc.sbc_count(h, 4, 3)]
        h.close()
        assert got == again == want


def test_failed_orientation_leaves_nothing(sbc):
    """A side whose build runs out of memory at its k-th block keeps no block of
    the failed call, and is built by the next one."""
    g = two_sided()
    want = oracle.count(g, 3, 4, side=0)
    for k in range(1, 20):
        with sbc.graph_from_synth(g) as h:
            held = sbc.sbc_graph_info(h)["device_bytes"]
            with RecordingAllocator(sbc, fail_at=k) as a:
                with pytest.raises(sbc.SbcError) as e:
                    sbc.sbc_count(h, 3, 4)
                assert e.value.status == 3  # SBC_E_NOMEM
                assert not a.live
            assert sbc.sbc_graph_info(h)["device_bytes"] == held
            assert sbc.sbc_count(h, 3, 4) == want


def test_batch_counts_again_after_a_failed_run(sbc, monkeypatch):
    """A run of a batch of several anchor groups plans again; when that runs out
    of memory at its k-th block, the next run is exact."""
    g = two_sided()
    want = oracle.count(g, 3, 3, side=0)
    monkeypatch.setenv("SBC_POOL_BUDGET_KB", "4")
    with RecordingAllocator(sbc) as a:
        with sbc.graph_from_synth(g) as h, sbc.Batch([h], 3, 3) as b:
            for k in range(1, 12):
                a.calls, a.fail_at = 0, k
                with pytest.raises(sbc.SbcError) as e:
                    b.run()
                assert e.value.status == 3  # SBC_E_NOMEM
                a.fail_at = 0
                assert b.run() == [want]
        assert not a.live
