"""The bucket path's producers (keys of a range appended a bufferful at a time,
edge ends of a range gathered by tiles) give the in-memory build's graph: with
one range and with many, at a few edges and around a tile of 2048, with reads
of one instance, and with nearly every key in one range."""
from __future__ import annotations

import numpy as np
import pytest

from parity import gpu_graph
from paper_1003_1940_gb300 import readgen

pytestmark = pytest.mark.gpu


def same(dbg, reads, lengths, k, budget):
    _, want = gpu_graph(dbg, dbg.Context(), reads, lengths, k)
    g = dbg.dbg_build_bucketed(dbg.Context(), reads, lengths, k, budget)
    got = {"nodes": dbg.dbg_graph_nodes(g), **{f"e_{a}": b for a, b in dbg.dbg_graph_edges(g).items()},
           **{f"c_{a}": b for a, b in dbg.dbg_graph_csr(g).items()}}
    for key, array in got.items():
        np.testing.assert_array_equal(array, want[key], err_msg=key)
    return dbg.dbg_graph_buckets(g), want


@pytest.mark.parametrize("k", [5, 21, 31, 33, 63])
@pytest.mark.parametrize("n,budget", [(1, 0), (40, 0), (6_000, 0), (6_000, 1 << 20), (40_000, 4 << 20)])
def test_ranges(k, n, budget):
    from paper_1003_1940_gb300 import dbg
    reads, _ = readgen.generate(readgen.ReadSetSpec(200_000, n, k + 45, 0.01, k, 7 + k))
    lengths = np.random.default_rng(n + k).integers(k - 2, k + 46, n).astype(np.uint32)
    lengths[0] = k + 45
    reads = np.concatenate([row[:m] for row, m in zip(reads.reshape(n, -1), lengths)])
    same(dbg, reads, lengths, k, budget)


@pytest.mark.parametrize("edges", [2047, 2048, 2049, 4096])
def test_tile_edges(edges):
    from paper_1003_1940_gb300 import dbg
    k = 31
    rng = np.random.default_rng(edges)
    read = np.frombuffer(b"ACGT", dtype=np.uint8)[rng.integers(0, 4, edges + k)]
    _, want = same(dbg, read, np.array([edges + k], dtype=np.uint32), k, 0)
    assert want["E"] == edges


def test_crowded_range():
    from paper_1003_1940_gb300 import dbg
    k = 21
    rng = np.random.default_rng(3)
    # poly-A heads put the keys of one instance per read under one prefix
    body = np.frombuffer(b"ACGT", dtype=np.uint8)[rng.integers(0, 4, (150_000, 10))]
    reads = np.concatenate([np.full((150_000, 12), ord("A"), dtype=np.uint8), body], axis=1).reshape(-1)
    ranges, _ = same(dbg, reads, np.full(150_000, 22, dtype=np.uint32), k, 2 << 20)
    assert ranges[0] >= 1
