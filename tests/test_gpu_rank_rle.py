"""Tiles of nearly distinct edge keys, ranked copy by copy: a read repeated up
to, at and past a bucket's limit (512 copies) and past a tile's capacity,
among reads that hold every key about once, gives the edge list of sorting
every copy by digits, and the oracle's."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from parity import assert_graph_equal, gpu_graph
from paper_1003_1940_gb300 import readgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [15, 31, 41])
@pytest.mark.parametrize("copies", [1, 2, 511, 513, 2000, 7000])
def test_repeats_among_distinct_keys(k, copies):
    from paper_1003_1940_gb300 import dbg
    L = k + 40
    reads, lengths = readgen.generate(readgen.ReadSetSpec(3_000_000, 1_500, L, 0.0, k, 17 + k))
    one = np.tile(reads[:L // 2 + k // 2 + 3], copies)
    reads = np.concatenate([reads, one])
    lengths = np.concatenate([lengths, np.full(copies, len(one) // copies, dtype=np.uint32)])
    got = []
    for count, rank in ((True, True), (True, False), (False, False)):
        ctx = dbg.Context()
        dbg.dbg_sort_count_first_set(ctx, count)
        dbg.dbg_sort_local_rank_set(ctx, rank)
        got.append(gpu_graph(dbg, ctx, reads, lengths, k)[1])
    for other in got[1:]:
        for key in got[0]:
            np.testing.assert_array_equal(got[0][key], other[key], err_msg=key)
    assert_graph_equal(got[0], oracle.build_graph(reads, lengths, k))
