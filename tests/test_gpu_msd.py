"""The sorts most significant digit first (unordered partition passes, then
the local pass) give bit for bit the graph of the ordered, least-significant-
first passes, of every digit sorted globally, and the oracle's: at the sizes
where the number of passes and the last tile change, for both key widths,
with reads of exactly k bases, with the distinct-read counts (records whose
payload order matters), and for keys crowded into few first digits."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from parity import assert_graph_equal, gpu_graph
from paper_1003_1940_gb300 import readgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dbg():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1003_1940_gb300 import dbg as d
    d.load()
    return d


def exact_instances(N: int, k: int, seed: int, genome: int):
    """Reads holding exactly N edge instances, and 20 of exactly k bases."""
    per = 50
    reads, lengths = readgen.generate(readgen.ReadSetSpec(genome, N // per + 21, k + per, 0.01, k, seed))
    parts = reads.reshape(-1, k + per)
    keep = [parts[i] for i in range(N // per)]
    tail = [parts[-1][:k + N % per]] if N % per else []
    iso = [p[:k] for p in parts[-21:-1]]
    rows = keep + tail + iso
    return np.concatenate(rows), np.array([len(r) for r in rows], dtype=np.uint32)


def ways(dbg, reads, lengths, k, with_oracle=True):
    """msd, ordered passes, ordered with digit-pass local sorts, all digits
    globally: graphs and distinct-read counts."""
    got = []
    for partition, rank, hybrid in ((True, True, True), (False, True, True), (True, False, True), (True, True, False)):
        ctx = dbg.Context()
        dbg.dbg_sort_partition_first_set(ctx, partition)
        dbg.dbg_sort_local_rank_set(ctx, rank)
        dbg.dbg_sort_hybrid_set(ctx, hybrid)
        dbg.dbg_node_reads_set(ctx, True)
        g, d = gpu_graph(dbg, ctx, reads, lengths, k)
        d["node_reads"] = dbg.dbg_graph_node_reads(g)
        got.append(d)
    for other in got[1:]:
        for key in got[0]:
            np.testing.assert_array_equal(got[0][key], other[key], err_msg=key)
    if with_oracle:
        assert_graph_equal(got[0], oracle.build_graph(reads, lengths, k))
        np.testing.assert_array_equal(got[0]["node_reads"], oracle.node_reads(reads, lengths, k)[1])


@pytest.mark.parametrize("k,N", [(31, 1), (31, 4096), (31, 4097), (31, 12289), (21, 1 << 20), (21, (1 << 20) + 1),
                                 (33, 2048), (33, 2049), (55, 1 << 19), (55, (1 << 19) + 1)])
def test_pass_counts(dbg, k, N):
    """One local tile, one pass, two passes."""
    ways(dbg, *exact_instances(N, k, 1000 + N % 97 + k, max(2_000, N // 8)), k)


@pytest.mark.parametrize("k,n", [(21, 4_000), (31, 40_000), (41, 20_000)])
def test_crowded_first_digits(dbg, k, n):
    """Reads of mostly A: nearly every key shares its first digits, so one
    bucket holds most keys, groups run far over the mean size and some over
    what a local tile holds."""
    rng = np.random.default_rng(k)
    L = k + 40
    reads = np.frombuffer(b"ACGT", dtype=np.uint8)[rng.choice(4, size=n * L, p=[0.91, 0.04, 0.03, 0.02])]
    ways(dbg, np.ascontiguousarray(reads), np.full(n, L, dtype=np.uint32), k)


@pytest.mark.parametrize("k", [5, 9, 11, 13])
def test_short_keys(dbg, k):
    """Few possible keys: too few for the partition passes (k = 5), or
    groups of a few key values with many copies each."""
    reads, lengths = readgen.generate(readgen.ReadSetSpec(60_000, 20_000, 100, 0.01, k, 1100 + k))
    ways(dbg, reads, lengths, k)
