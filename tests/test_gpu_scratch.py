"""Results do not live in a context's scratch block: graphs and unitigs of one
context, at sizes below and above the block's largest piece and with tandem
repeats (oversize tiles) among them, stay what a fresh context gives while
the context goes on building."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1003_1940_gb300 import readgen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("torch_allocator", [True, False])
def test_results_outlive_scratch(torch_allocator):
    from paper_1003_1940_gb300 import dbg
    sets = []
    for seed, (reads, genome) in enumerate([(3, 200), (400, 3000), (60_000, 300_000), (7, 90), (9_000, 400_000)]):
        bases, lengths = readgen.generate(readgen.ReadSetSpec(genome, reads, 60, 0.01, 21, seed))
        if seed % 2:  # 20 kbp of one unit of three bases
            unit = np.tile(np.frombuffer(b"ACG", dtype=np.uint8), 7000).astype(bases.dtype)
            bases, lengths = np.concatenate([bases, unit]), np.append(lengths, np.uint32(len(unit)))
        sets.append((bases, lengths))
    def read(g, u):
        return {"nodes": dbg.dbg_graph_nodes(g), **dbg.dbg_graph_edges(g), **dbg.dbg_graph_csr(g),
                **{f"u_{a}": np.asarray(b) for a, b in dbg.dbg_unitigs_get(u).items()}}

    ctx = dbg.Context(torch_allocator=torch_allocator)
    kept = []
    for bases, lengths in sets + sets[:2]:
        g = dbg.dbg_build(ctx, bases, lengths, 21)
        kept.append((g, dbg.dbg_compact(ctx, g)))
    for (g, u), (bases, lengths) in zip(kept, sets + sets[:2]):
        other = dbg.Context(torch_allocator=torch_allocator)
        want = dbg.dbg_build(other, bases, lengths, 21)
        expected = read(want, dbg.dbg_compact(other, want))
        for key, array in read(g, u).items():
            np.testing.assert_array_equal(array, expected[key], err_msg=key)
