"""The context's scratch block and memory that runs short: a call that fits
without the block fits with it (the block goes back and the call is made
again), a context that met a shortage holds no block afterwards, and calls
within a memory budget, and idle server workers, hold little or nothing."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

from paper_1003_1940_gb300 import readgen

pytestmark = pytest.mark.gpu

BLOCK = 32 << 20


class Counted:
    """Device memory through the library's hooks, counted and limited."""

    def __init__(self, dbg, limit=1 << 60):
        import torch
        self.limit, self.live, self.peak, self.refused = limit, 0, 0, 0
        self.largest, self.seen = 1 << 60, set()  # of one allocation: the most allowed; the sizes seen
        self.sizes = {}

        def alloc(user, nbytes, stream):
            if self.live + nbytes > self.limit or nbytes > self.largest:
                self.refused += 1
                return None
            p = int(torch.cuda.caching_allocator_alloc(int(nbytes), 0, stream or 0))
            self.sizes[p] = nbytes
            self.seen.add(nbytes)
            self.live += nbytes
            self.peak = max(self.peak, self.live)
            return p

        def free(user, ptr, nbytes, stream):
            self.live -= self.sizes.pop(ptr)
            torch.cuda.caching_allocator_delete(ptr)

        self.hooks = dbg._ALLOC_FN(alloc), dbg._FREE_FN(free)
        ctx = dbg.Context(device=0)
        ctx.close()
        opt = ctx._opt
        opt.alloc, opt.free = self.hooks
        h = ctypes.c_void_p()
        dbg._check(dbg.load().dbg_create(ctypes.byref(h), ctypes.byref(opt)), "dbg_create")
        ctx.handle = h
        ctx._hooks = self
        self.ctx = ctx


@pytest.fixture(scope="module")
def data():
    return readgen.generate(readgen.ReadSetSpec(200_000, 40_000, 60, 0.01, 31, 4))


def graph_of(dbg, g):
    return {"nodes": dbg.dbg_graph_nodes(g), **dbg.dbg_graph_edges(g), **dbg.dbg_graph_csr(g)}


def test_call_that_fits_without_the_block(data):
    from paper_1003_1940_gb300 import dbg
    reads, lengths = data

    def calls(ctx):
        g = dbg.dbg_build(ctx, reads, lengths, 31)
        return g, dbg.dbg_compact(ctx, g), dbg.dbg_simplify(ctx, g, 3)

    free = Counted(dbg, limit=0)  # the first allocation fails: no block from then on
    with pytest.raises(dbg.DbgError, match="ENOMEM"):
        dbg.dbg_build(free.ctx, reads, lengths, 31)
    free.limit = 1 << 60
    want = calls(free.ctx)
    expected = graph_of(dbg, want[0])
    need = free.peak

    tight = Counted(dbg, limit=need)
    got = calls(tight.ctx)
    assert tight.refused > 0
    for key, array in graph_of(dbg, got[0]).items():
        np.testing.assert_array_equal(array, expected[key], err_msg=key)
    for key, array in dbg.dbg_unitigs_get(got[1]).items():
        assert np.array_equal(np.asarray(array), np.asarray(dbg.dbg_unitigs_get(want[1])[key])), key
    del got
    assert tight.live == 0  # nothing held once a shortage was met


def test_block_is_kept_and_given_back(data):
    from paper_1003_1940_gb300 import dbg
    reads, lengths = data
    hooks = Counted(dbg)
    g = dbg.dbg_build(hooks.ctx, reads, lengths, 31)
    del g
    assert hooks.live == BLOCK
    hooks.limit = hooks.live + 1000  # the next build runs short in the middle
    with pytest.raises(dbg.DbgError, match="ENOMEM"):
        dbg.dbg_build(hooks.ctx, reads, lengths, 31)
    assert hooks.live == 0
    hooks.ctx.close()


@pytest.mark.parametrize("budget_mb", [1, 16, 64])
def test_budgeted_call(data, budget_mb):
    """The block of a call within a budget is at most a sixteenth of it (or
    256 KB), whatever the context held before, and goes back with the call."""
    from paper_1003_1940_gb300 import dbg
    reads, lengths = data
    hooks = Counted(dbg)
    g = dbg.dbg_build(hooks.ctx, reads, lengths, 31)
    want = graph_of(dbg, g)
    del g
    assert hooks.live == BLOCK
    before = set(hooks.sizes)
    g = dbg.dbg_build_bucketed(hooks.ctx, reads, lengths, 31, budget_mb << 20)
    assert not before & set(hooks.sizes)  # the large block went back
    for key, array in graph_of(dbg, g).items():
        np.testing.assert_array_equal(array, want[key], err_msg=key)
    del g
    assert hooks.live == 0
    dbg.dbg_build(hooks.ctx, reads, lengths, 31)
    assert hooks.live == BLOCK  # and the next call has its own again


@pytest.mark.parametrize("k", [31, 41])
def test_arrays_one_by_one(data, k):
    """Memory that has room for every array but not for several in one piece:
    the graph's arrays are then allocations of their own."""
    from paper_1003_1940_gb300 import dbg
    reads, lengths = data
    hooks = Counted(dbg)
    g = dbg.dbg_build(hooks.ctx, reads, lengths, k)
    want = graph_of(dbg, g)
    other = Counted(dbg)
    other.largest = max(n for n in hooks.seen if n != BLOCK) - 1
    h = dbg.dbg_build(other.ctx, reads, lengths, k)
    for key, array in graph_of(dbg, h).items():
        np.testing.assert_array_equal(array, want[key], err_msg=key)
    assert other.refused > 0
    other.largest = 1 << 60
    u, v = dbg.dbg_unitigs_get(dbg.dbg_compact(hooks.ctx, g)), dbg.dbg_unitigs_get(dbg.dbg_compact(other.ctx, h))
    for key in u:
        assert np.array_equal(np.asarray(u[key]), np.asarray(v[key])), key
    del h, v
    assert other.live in (0, BLOCK)


@pytest.mark.parametrize("k", [31, 55])
def test_counts_hold_no_staged_multiplicities(k):
    """The most device memory of a build with both counts, itemised: the k-mer
    sort beside the distinct edge keys' buffer and one multiplicity per edge,
    not per instance."""
    from paper_1003_1940_gb300 import dbg
    n, L, w = 200_000, 100, 8 if k <= 31 else 16
    reads, lengths = readgen.generate(readgen.ReadSetSpec(n * L // 30, n, L, 0.002, k, 8))
    hooks = Counted(dbg)
    dbg.dbg_node_mult_set(hooks.ctx, True)
    dbg.dbg_node_reads_set(hooks.ctx, True)
    g = dbg.dbg_build(hooks.ctx, reads, lengths, k)
    N, M, E, V = n * (L - k), n * (L - k + 1), dbg.dbg_graph_num_edges(g), dbg.dbg_graph_num_nodes(g)
    held = N * w + 4 * E + 4 * V + n * L // 4 + 24 * n
    sort = M * (2 * w + 8) + 12 * M
    tables = M // 4 + (2 << 20)
    assert hooks.peak <= BLOCK + held + sort + tables, (hooks.peak, held, sort)


def test_idle_workers_hold_nothing(data):
    """Device memory after a server has been idle for a while is what it was
    before its workers built anything (its contexts take cudaMallocAsync memory:
    the pool's bytes in use are looked at)."""
    import time

    import torch
    from paper_1003_1940_gb300 import dbg
    reads, lengths = data

    def in_use():
        torch.cuda.synchronize()
        cudart = ctypes.CDLL(None)
        pool, used = ctypes.c_void_p(), ctypes.c_uint64()
        get, attr = cudart.cudaDeviceGetDefaultMemPool, cudart.cudaMemPoolGetAttribute
        assert get(ctypes.byref(pool), 0) == 0 and attr(pool, 7, ctypes.byref(used)) == 0  # UsedMemCurrent
        return used.value

    srv = dbg.Server(workers=3)
    before = in_use()
    tickets = [dbg.dbg_submit(srv, reads, lengths, 31) for _ in range(6)]
    for t in tickets:
        g, _ = dbg.dbg_poll(srv, t)
        g.free()
    time.sleep(0.1)
    held = in_use() - before
    srv.close()
    assert held < BLOCK  # (the look-back words of each context stay)
