"""Genomes of uneven base composition, whose AT-rich prefixes put many keys into
few groups: the groups that are too long for a local tile are split, and the
graph and the counts are those of the ordered passes -- at sizes of one and of
two partition passes, for both key widths, with the count-first pass on and
off, with reads of exactly k bases, in the bucket path, and with the copies of
one k-mer (which no split divides) among the long groups."""
from __future__ import annotations

import numpy as np
import pytest

from parity import gpu_graph

pytestmark = pytest.mark.gpu


def read_set(n, L, gc, k, hot, seed):
    rng = np.random.default_rng(seed)
    p = [(1 - gc) / 2, gc / 2, gc / 2, (1 - gc) / 2]
    genome = rng.choice(4, size=max(2_000, n * L // 12), p=p).astype(np.uint8)
    rows = genome[rng.integers(0, len(genome) - L + 1, n)[:, None] + np.arange(L)]
    back = rng.random(n) < 0.5
    rows[back] = 3 - rows[back, ::-1]
    hit = rng.random(rows.shape) < 0.005
    rows[hit] = (rows[hit] + rng.integers(1, 4, int(hit.sum()))) & 3
    if hot:  # a share of the reads is one base, or one unit of three
        rows[: int(hot * n)] = 0
        rows[int(hot * n): int(1.5 * hot * n)] = np.resize(np.array([0, 1, 3], dtype=np.uint8), L)
    lengths = np.full(n, L, dtype=np.uint32)
    lengths[5::97] = k
    keep = np.arange(L)[None, :] < lengths[:, None]
    return np.frombuffer(b"ACGT", dtype=np.uint8)[rows[keep]], lengths


def build(dbg, reads, lengths, k, partition=True, count=True, rank=True):
    ctx = dbg.Context()
    dbg.dbg_sort_partition_first_set(ctx, partition)
    dbg.dbg_sort_count_first_set(ctx, count)
    dbg.dbg_sort_local_rank_set(ctx, rank)
    dbg.dbg_node_mult_set(ctx, True)
    dbg.dbg_node_reads_set(ctx, True)
    g, d = gpu_graph(dbg, ctx, reads, lengths, k)
    d["node_mult"], d["node_reads"] = dbg.dbg_graph_node_mult(g), dbg.dbg_graph_node_reads(g)
    return d, dbg.dbg_sort_fallbacks(ctx)


@pytest.mark.parametrize("k,n,gc,hot", [(31, 9_300, 0.2, 0.0), (31, 9_300, 0.33, 0.0), (21, 9_300, 0.2, 0.1),
                                        (41, 9_300, 0.2, 0.0), (31, 60_000, 0.2, 0.0), (31, 60_000, 0.2, 0.3),
                                        (55, 60_000, 0.15, 0.05), (13, 40_000, 0.2, 0.0)])
def test_splits(k, n, gc, hot):
    from paper_1003_1940_gb300 import dbg
    reads, lengths = read_set(n, 100, gc, k, hot, k + n)
    want, _ = build(dbg, reads, lengths, k, partition=False)
    for switches in ({}, {"count": False}, {"rank": False}):
        got, _ = build(dbg, reads, lengths, k, **switches)
        for key in want:
            np.testing.assert_array_equal(got[key], want[key], err_msg=f"{key} {switches}")
    g = dbg.dbg_build_bucketed(dbg.Context(), reads, lengths, k, 24 << 20)
    for key, array in dbg.dbg_graph_edges(g).items():
        np.testing.assert_array_equal(array, want[f"e_{key}"], err_msg=key)
    for key, array in dbg.dbg_graph_csr(g).items():
        np.testing.assert_array_equal(array, want[f"c_{key}"], err_msg=key)


@pytest.mark.parametrize("n", [9_300, 60_000])
def test_no_sort_over_every_digit(n):
    """At 20 % GC every third key is in a long group; split, none of them is
    left to the sort over every digit."""
    from paper_1003_1940_gb300 import dbg
    reads, lengths = read_set(n, 100, 0.2, 31, 0.0, 9)
    ctx = dbg.Context()
    dbg.dbg_build(ctx, reads, lengths, 31)
    assert dbg.dbg_sort_fallbacks(ctx) == 0
