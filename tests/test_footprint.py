"""The admission footprint of a build bounds what the build holds at its
fullest points, itemised here buffer by buffer, when every key is distinct and
every record lies in a tile too long for shared memory: both key widths."""
from __future__ import annotations

import ctypes

import pytest

from paper_1003_1940_gb300 import build_lib


@pytest.mark.parametrize("k", [21, 31, 33, 63])
@pytest.mark.parametrize("N,I,n", [(0, 0, 0), (10_000, 0, 100), (50_000_000, 10, 700_000), (3_000_000_000, 0, 30_000_000),
                                   (1_000_000, 40_000_000, 41_000_000)])
def test_bounds_every_stage(k, N, I, n):
    f = ctypes.CDLL(build_lib.build())._ZN3dbg15build_footprintEmmmmjbb
    f.restype = ctypes.c_uint64
    f.argtypes = [ctypes.c_uint64] * 4 + [ctypes.c_uint32, ctypes.c_bool, ctypes.c_bool]
    w = 8 if k <= 31 else 16
    bases = N + n * k + I
    got = f(n, bases, N, I, k, False, False)
    E, R = N, 2 * N + I
    reads = 16 * (n + 1) + bases // 4
    tile, cap_mean = (4096, 1024) if w == 8 else (2048, 512)

    def tables(keys):  # of a sort: tiles, groups, and the parts of split groups
        return 52 * (keys // tile + 1) + 12 * (2 * keys // cap_mean) + 12 * (2 * keys // (tile // 16))

    keys = {"buffers": 2 * N * w, "staged counts": 4 * N, "gathered": 2 * N * w, "distinct": N * w, "heads": 4 * N}
    edges = {"edge arrays": E * (w + 4 + 1)}
    records = {"buffers": 2 * R * (w + 4), "heads": R // 8}
    gather = {"gathered": R * (w + 4), "words": 16 * R, "permuted": R * (w + 4)}
    stages = [
        sum(keys.values()) + tables(N),
        N * w + 4 * N + sum(edges.values()) + R * (w + 4),  # edge ends: staged keys and counts, one record buffer
        sum(edges.values()) + sum(records.values()) + sum(gather.values()) + tables(R),
        # the node-ID pass
        sum(edges.values()) + sum(records.values()) + tables(R) + R * w + 8 * (R + 1) + 8 * E + (8 + 8 + 2 + 2) * E + 16 * E,
    ]
    assert got >= reads + max(stages), [x / max(1, N) for x in (got, *stages)]
