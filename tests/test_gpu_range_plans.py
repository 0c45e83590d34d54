"""The bucket path plans each range's sort over the range: with many key ranges
of a uniform genome, no local tile is longer than shared memory holds (the
fallback counter stays at 0), the ranges number what the budget asks for, and
the graph is the in-memory build's.  Reads of exactly k bases are among them.
Keys of few bits, whose ranges are single key values, come out right too."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1003_1940_gb300 import readgen

pytestmark = pytest.mark.gpu


def compare(dbg, ctx, reads, lengths, k, budget):
    want = dbg.dbg_build(dbg.Context(), reads, lengths, k)
    g = dbg.dbg_build_bucketed(ctx, reads, lengths, k, budget)
    for a, b in ((dbg.dbg_graph_edges(g), dbg.dbg_graph_edges(want)), (dbg.dbg_graph_csr(g), dbg.dbg_graph_csr(want)),
                 ({"nodes": dbg.dbg_graph_nodes(g)}, {"nodes": dbg.dbg_graph_nodes(want)})):
        for key in a:
            np.testing.assert_array_equal(a[key], b[key], err_msg=key)
    return dbg.dbg_graph_buckets(g)


@pytest.mark.parametrize("partition", [True, False])
@pytest.mark.parametrize("k,budget_mb,edges,nodes", [(31, 60, 3, 9), (31, 22, 9, 20), (31, 12, 20, 20), (55, 60, 4, 20),
                                                     (55, 24, 9, 20), (33, 24, 9, 20)])
def test_many_ranges(k, budget_mb, edges, nodes, partition):
    from paper_1003_1940_gb300 import dbg
    n = 100_000 if k < 40 else 160_000
    reads, lengths = readgen.generate(readgen.ReadSetSpec(n * 100 // 30, n, 100, 0.005, k, 11))
    lengths = lengths.copy()
    lengths[::1000] = k  # reads of one k-mer and no edge
    keep = np.arange(100)[None, :] < lengths[:, None]
    reads = reads.reshape(n, 100)[keep]
    ctx = dbg.Context()
    dbg.dbg_sort_partition_first_set(ctx, partition)
    ranges = compare(dbg, ctx, reads, lengths, k, budget_mb << 20)
    assert ranges[0] >= edges and ranges[1] >= nodes, ranges
    assert dbg.dbg_sort_fallbacks(ctx) == 0


@pytest.mark.parametrize("k", [1, 3, 5, 7])
def test_short_keys(k):
    from paper_1003_1940_gb300 import dbg
    reads, lengths = readgen.generate(readgen.ReadSetSpec(20_000, 4_000, 60, 0.01, k, 3))
    ranges = compare(dbg, dbg.Context(), reads, lengths, k, 1 << 20)
    assert ranges[0] > 1 if k >= 5 else ranges[0] >= 1
