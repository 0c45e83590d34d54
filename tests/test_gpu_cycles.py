"""Circular chains of all sizes, alone, beside short chains (the walks finish
and the cycles are ranked apart), beside long ones (ranked by segments), and
with branches into other circles: every mode gives the oracle's unitigs, and
so does the simplified graph."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from parity import assert_unitigs_equal

pytestmark = pytest.mark.gpu

FIELDS = ("node_off", "nodes", "seq_off", "circular")


def bases(rng, n):
    return np.frombuffer(b"ACGT", dtype=np.uint8)[rng.integers(0, 4, size=n)]


def circle(rng, n, k):
    c = bases(rng, n)
    return np.resize(c, n + k)


def check(reads, k):
    from paper_1003_1940_gb300 import dbg
    lengths = np.array([len(r) for r in reads], dtype=np.uint32)
    data = np.concatenate(reads)
    ctx = dbg.Context()
    g = dbg.dbg_build(ctx, data, lengths, k)
    want = oracle.compact(oracle.build_graph(data, lengths, k))
    simple = []
    for mode in (0, 1, 2):
        dbg.dbg_compact_mode_set(ctx, mode)
        u = dbg.dbg_unitigs_get(dbg.dbg_compact(ctx, g))
        assert_unitigs_equal(u, want)
        simple.append(dbg.dbg_simple_get(dbg.dbg_simplify(ctx, g, 3)))
    for other in simple[1:]:
        for key in simple[0]:
            assert np.array_equal(np.asarray(other[key]), np.asarray(simple[0][key])), key
    return u


@pytest.mark.parametrize("k", [21, 33])
@pytest.mark.parametrize("sizes", [(2,), (3,), (50, 51, 7), (900, 5_000, 4), tuple(range(2, 130, 3))])
def test_only_circles(k, sizes):
    rng = np.random.default_rng(sum(sizes) + k)
    u = check([circle(rng, n, k) for n in sizes], k)
    assert int(u["circular"].sum()) >= len(sizes) // 2


@pytest.mark.parametrize("k", [21, 41])
@pytest.mark.parametrize("sizes", [(5_000,), (2, 33, 64, 700, 3_001), tuple(range(4, 300, 7))])
def test_beside_short_lists(k, sizes):
    """Thousands of short chains of reads around the circles."""
    rng = np.random.default_rng(len(sizes) + k)
    reads = [bases(rng, k + int(x)) for x in rng.integers(0, 60, 3_000)]
    for i, n in enumerate(sizes):
        reads.insert(1 + 7 * i, circle(rng, n, k))
    u = check(reads, k)
    assert int(u["circular"].sum()) >= len(sizes) // 2


@pytest.mark.parametrize("k", [21, 33])
@pytest.mark.parametrize("lists,sizes", [(1, (3,)), (2, (3, 40, 6_000)), (2, (9_000,)), (30, (100, 20_000))])
def test_beside_long_lists(k, lists, sizes):
    rng = np.random.default_rng(lists + k)
    u = check([bases(rng, 20_000) for _ in range(lists)] + [circle(rng, n, k) for n in sizes], k)
    assert int(u["circular"].sum()) >= 1


def test_circles_that_share_a_stretch():
    """Two circles through the same 200 bases: chains between branches, and
    one circle beside them that keeps whole."""
    k = 21
    rng = np.random.default_rng(1)
    shared = bases(rng, 200)
    reads = []
    for n in (700, 900):
        c = np.concatenate([shared, bases(rng, n)])
        reads.append(np.resize(c, len(c) + k))
    reads += [circle(rng, 1_234, k), bases(rng, 500)]
    u = check(reads, k)
    assert int(u["circular"].sum()) == 1


@pytest.mark.parametrize("long_lists", [False, True])
def test_links_are_made_once(long_lists):
    """A circle among the chains does not send the graph through the link
    kernels again (two launches; with long lists one more, which takes the
    successors from what they made)."""
    from paper_1003_1940_gb300 import dbg
    k = 21
    rng = np.random.default_rng(3)
    reads = [circle(rng, 500, k)] + [bases(rng, 30_000 if long_lists else 60) for _ in range(2 if long_lists else 3_000)]
    ctx = dbg.Context()
    g = dbg.dbg_build(ctx, np.concatenate(reads), np.array([len(r) for r in reads], dtype=np.uint32), k)
    dbg.dbg_profile_enable(ctx, True)
    u = dbg.dbg_unitigs_get(dbg.dbg_compact(ctx, g))
    assert int(u["circular"].sum()) == 1
    assert dbg.dbg_profile_read(ctx)["compact_links"]["launches"] == (3 if long_lists else 2)
