"""Compaction of graphs with few, long lists, which are ranked by segments
(modes 0 and 1) instead of the meeting walks: the unitigs of pointer jumping
alone (mode 2) and the oracle's -- one list, many lists on both sides of what
a pair of walkers may take (4096 nodes), lists with branches between them,
and a cycle beside long lists, with and without a splitter on it."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from parity import assert_unitigs_equal

pytestmark = pytest.mark.gpu

FIELDS = ("node_off", "nodes", "seq_off", "circular")


@pytest.fixture(scope="module")
def dbg():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1003_1940_gb300 import dbg as d
    d.load()
    return d


def check(dbg, reads, k):
    lengths = np.array([len(r) for r in reads], dtype=np.uint32)
    data = np.concatenate(reads)
    ctx = dbg.Context()
    g = dbg.dbg_build(ctx, data, lengths, k)
    got = []
    for mode in (0, 1, 2):
        dbg.dbg_compact_mode_set(ctx, mode)
        got.append(dbg.dbg_unitigs_get(dbg.dbg_compact(ctx, g)))
    for other in got[1:]:
        for f in FIELDS:
            np.testing.assert_array_equal(other[f], got[0][f], err_msg=f)
        assert other["seq"] == got[0]["seq"]
    assert_unitigs_equal(got[0], oracle.compact(oracle.build_graph(data, lengths, k)))
    return got[0]


def genome(rng, n):
    return np.frombuffer(b"ACGT", dtype=np.uint8)[rng.integers(0, 4, size=n)]


@pytest.mark.parametrize("k", [21, 33])
@pytest.mark.parametrize("lists,length", [(1, 60), (1, 5_000), (1, 60_000), (40, 4_096), (40, 4_200), (300, 900),
                                          (2, 100_003)])
def test_long_lists(dbg, k, lists, length):
    rng = np.random.default_rng(lists * 7 + length + k)
    u = check(dbg, [genome(rng, length + k - 1) for _ in range(lists)], k)
    assert len(u["circular"]) == lists and int(np.diff(u["node_off"]).max()) == length


@pytest.mark.parametrize("k", [21, 41])
def test_branches_between_long_lists(dbg, k):
    """Repeats of more than k bases shared by long sequences."""
    rng = np.random.default_rng(k)
    rep = [genome(rng, 200) for _ in range(3)]
    reads = []
    for i in range(12):
        reads.append(np.concatenate([genome(rng, 3_000 + 500 * i), rep[i % 3], genome(rng, 2_000)]))
    u = check(dbg, reads, k)
    assert len(u["circular"]) > 12


@pytest.mark.parametrize("circle", [4, 9, 700, 6_000])
def test_cycle_beside_long_lists(dbg, circle):
    k = 21
    rng = np.random.default_rng(circle)
    c = genome(rng, circle)
    wrapped = np.resize(c, circle + k)
    u = check(dbg, [genome(rng, 30_000), wrapped, genome(rng, 9_000)], k)
    assert int(u["circular"].sum()) == 1
