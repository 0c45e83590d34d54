"""Local tiles that hold copies of one key only, in groups with no key bits
left below them (k = 7: 16-bit edge keys and 16 M instances of an uneven
composition, so that the densest buckets resolve every bit, with some 4500
copies of each of their keys): the digit-pass kernels sort and count them like
any other tile, with the count-first pass off and on."""
from __future__ import annotations

import numpy as np
import pytest

from parity import gpu_graph

pytestmark = pytest.mark.gpu


def test_tiles_of_one_key():
    from paper_1003_1940_gb300 import dbg
    k, n, L = 7, 160_000, 107
    rng = np.random.default_rng(7)
    reads = np.frombuffer(b"ACGT", dtype=np.uint8)[rng.choice(4, size=n * L, p=[0.33, 0.17, 0.17, 0.33])]
    lengths = np.full(n, L, dtype=np.uint32)
    got = []
    for hybrid, count, rank in ((False, True, True), (True, False, True), (True, False, False), (True, True, False),
                                (True, True, True)):
        ctx = dbg.Context()
        dbg.dbg_sort_hybrid_set(ctx, hybrid)
        dbg.dbg_sort_count_first_set(ctx, count)
        dbg.dbg_sort_local_rank_set(ctx, rank)
        dbg.dbg_node_mult_set(ctx, True)
        g, d = gpu_graph(dbg, ctx, reads, lengths, k)
        d["node_mult"] = dbg.dbg_graph_node_mult(g)
        got.append(d)
    mult = got[0]["e_mult"]
    assert np.count_nonzero((mult > 4096) & (mult <= 6144)) >= 50
    for other in got[1:]:
        for key in got[0]:
            np.testing.assert_array_equal(got[0][key], other[key], err_msg=key)
