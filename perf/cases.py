"""The work that users of this framework have it do, as cases to measure.

A case is one call sequence through the public entry points
(paper_1003_1940_gb300.dbg) on seeded synthetic sequencing reads:

  build          dbg_build of reads in device memory
  build_compact  dbg_build, then dbg_compact of the graph
  compact        dbg_compact of a graph already in hand
  simplify       dbg_simplify of a graph already in hand, read back
  counts         dbg_build with node multiplicities and roadmap counts on
  batch          dbg_build_batch of six read sets of uneven sizes
  host           pinned host reads in, the whole graph and its unitigs out
                 into pinned host buffers
  bucketed       dbg_build_bucketed within a device-memory budget

Results are read through the accessors into buffers that the program keeps
(device memory, pinned host memory or numpy arrays), sized before the data
are known; what lies behind a result stays zero.

The read sets follow the recipes of paper_1003_1940_gb300/readgen.py (genome,
repeat families, tandem arrays, both strands, substitution errors), drawn on
the GPU.  Every output is an integer array (keys, IDs, offsets, counts,
flags, ASCII), so outputs are exact and `exact` has nothing to add.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1003_1940_gb300 import dbg

# (field, entries, element type, W words per entry)
GRAPH_FIELDS = (("node_keys", "V", torch.int64, True), ("edge_keys", "E", torch.int64, True),
                ("row_ptr", "V1", torch.int64, False), ("src", "E", torch.int32, False),
                ("dst", "E", torch.int32, False), ("mult", "E", torch.int32, False),
                ("adj_nbr", "E2", torch.int32, False), ("adj_edge", "E2", torch.int32, False),
                ("orient", "E", torch.uint8, False), ("adj_role", "E2", torch.uint8, False))


def _case(kind, k, reads, read_len, genome, err, min_len=0, repeats=0.0, tandem=0.0, tuned=False, budget_mb=0):
    """min_len > 0: read lengths uniform on [min_len, read_len]; tuned: the
    program calls dbg_autotune once, as bench.py does."""
    return {"kind": kind, "k": k, "reads": reads, "read_len": read_len, "min_len": min_len, "genome": genome,
            "err": err, "repeats": repeats, "tandem": tandem, "tuned": tuned, "budget_mb": budget_mb}


def listed():
    return [
        # the smallest request: a gene-sized contig's reads; launches and host work decide
        dict(_case("build", 21, 500, 36, 3_000, 0.01), name="build_500x36_k21"),
        # the tiny workload (10,000 reads of 36 bp, k = 21), graph and unitigs
        dict(_case("build_compact", 21, 10_000, 36, 100_000, 0.01), name="tiny_10kx36_k21"),
        # a bacterial-plasmid-sized set from the middle of the batched workload's range
        dict(_case("build", 21, 400_000, 75, 1_000_000, 0.005), name="build_400kx75_k21"),
        # trimmed reads of many lengths at low coverage: 128-bit keys, nearly every key distinct, reads of length <= k
        dict(_case("build", 41, 300_000, 250, 20_000_000, 0.01, min_len=20), name="ragged_300k_k41"),
        # the large workload at its full size, graph and unitigs (the headline)
        dict(_case("build_compact", 31, 15_000_000, 100, 50_000_000, 0.005, repeats=0.02, tuned=True),
             name="large_15Mx100_k31"),
        # the long-k workload at its full size: 128-bit keys, tandem repeats
        dict(_case("build_compact", 55, 4_000_000, 150, 20_000_000, 0.003, repeats=0.02, tandem=0.005, tuned=True),
             name="long_k_4Mx150_k55"),
        # compaction alone of a graph kept on the device (a tenth of the large workload)
        dict(_case("compact", 31, 1_500_000, 100, 5_000_000, 0.005, repeats=0.02), name="compact_1.5Mx100_k31"),
        # the simplified graph, read back by the host
        dict(_case("simplify", 31, 100_000, 100, 300_000, 0.005), name="simplify_100kx100_k31"),
        # VELVET-style roadmap counts beside the graph
        dict(_case("counts", 25, 1_000_000, 100, 4_000_000, 0.005), name="counts_1Mx100_k25"),
        # six read sets of uneven sizes at once
        dict(_case("batch", 31, 600_000, 100, 2_000_000, 0.005), name="batch_6sets_600kx100"),
        # a host program: pinned reads in, the whole result out
        dict(_case("host", 31, 1_500_000, 100, 5_000_000, 0.005, repeats=0.02), name="host_1.5Mx100_k31"),
        # the out-of-core construction: edge keys in several ranges
        dict(_case("bucketed", 31, 1_000_000, 100, 3_500_000, 0.005, budget_mb=700), name="bucketed_1Mx100_k31"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["build", "build", "build", "build_compact", "build_compact", "compact", "simplify", "counts",
                       "batch", "host", "bucketed"])
    top = {"build": 6_000_000, "build_compact": 6_000_000, "compact": 3_000_000, "simplify": 200_000,
           "counts": 1_200_000, "batch": 1_500_000, "host": 1_500_000, "bucketed": 1_500_000}[kind]
    reads = _log(rng, 20_000 if kind == "bucketed" else 300, top)
    read_len = rng.choice([36, 50, 75, 100, 125, 150, 251])
    k = rng.choice([k for k in (15, 17, 21, 25, 27, 31, 33, 41, 55, 63) if k < read_len - 4])
    if kind == "batch":
        k = 31 if read_len > 36 else 21
    min_len = rng.choice([0, 0, max(5, read_len // 8)])
    coverage = math.exp(rng.uniform(math.log(0.5), math.log(60.0)))
    genome = max(2_000, int(reads * read_len / coverage))
    # repeat families of up to 5 kbp (10 of them, 20 copies each) need a genome that holds them
    repeats = rng.choice([0.0, 0.02]) if genome >= 2_000_000 else 0.0
    err = rng.choice([0.0, 0.003, 0.005, 0.01])
    # no more than the large workload costs: at low coverage nearly every key is distinct
    while reads * read_len > 500_000_000 or min(reads * read_len, genome + reads * read_len * err * k) > 120_000_000:
        reads, genome = reads // 2, max(2_000, genome // 2)
    case = _case(kind, k, reads, read_len, genome, err, min_len=min_len, repeats=repeats, tuned=rng.random() < 0.5)
    if kind == "bucketed":  # room for the graph and for a part of the keys or records
        _, N, _, E, _, _ = _shape(case, reads, genome, k)
        case["budget_mb"] = 8 + int((E * 60 + (N * 24 + E * 80) * rng.uniform(0.1, 0.5)) * (1 if k <= 31 else 2) / 1e6)
    return case


# --------------------------------------------------------------------------
# read sets
# --------------------------------------------------------------------------
def _genome(case, genome_len, gen, rng):
    g = torch.randint(0, 4, (genome_len,), generator=gen, device="cuda", dtype=torch.uint8)
    pieces = []
    if case["repeats"] > 0:  # copies of ten families, 1 % diverged
        fams = [torch.randint(0, 4, (int(rng.integers(1000, 5001)),), generator=gen, device="cuda", dtype=torch.uint8)
                for _ in range(10)]
        covered, i = 0, 0
        while (i < 200 or covered < case["repeats"] * genome_len) and covered < 0.5 * genome_len:
            pieces.append(fams[i % 10])
            covered += pieces[-1].numel()
            i += 1
    if case["tandem"] > 0:
        covered = 0
        while covered < case["tandem"] * genome_len:
            unit, length = int(rng.integers(2, 101)), int(rng.integers(500, 5001))
            u = torch.randint(0, 4, (unit,), generator=gen, device="cuda", dtype=torch.uint8)
            pieces.append(u.repeat(-(-length // unit))[:length])
            covered += length
    if pieces:
        seg = genome_len // len(pieces)
        for slot, idx in enumerate(rng.permutation(len(pieces))):
            p = pieces[idx]
            if p.numel() >= seg:
                continue
            hit = torch.rand(p.numel(), generator=gen, device="cuda") < 0.01
            shift = torch.randint(1, 4, (p.numel(),), generator=gen, device="cuda", dtype=torch.uint8)
            at = slot * seg + int(rng.integers(0, seg - p.numel() + 1))
            g[at:at + p.numel()] = torch.where(hit, (p + shift) & 3, p)
    return g


def _reads(case, n, genome_len, seed):
    """(ASCII reads, int32 lengths), on the GPU."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rng = np.random.default_rng(seed)
    L, lo = case["read_len"], case["min_len"]
    genome = _genome(case, max(genome_len, L + 1), gen, rng)
    acgt = torch.tensor(list(b"ACGT"), device="cuda", dtype=torch.uint8)
    span = torch.arange(L, device="cuda")
    if lo:
        lengths = torch.randint(lo, L + 1, (n,), generator=gen, device="cuda", dtype=torch.int32)
    else:
        lengths = torch.full((n,), L, device="cuda", dtype=torch.int32)
    parts, step = [], max(1, (1 << 26) // L)
    for c in range(0, n, step):
        m = min(step, n - c)
        starts = torch.randint(0, genome.numel() - L + 1, (m, 1), generator=gen, device="cuda")
        block = genome[starts + span]
        back = torch.rand((m, 1), generator=gen, device="cuda") < 0.5
        block = torch.where(back, 3 - block.flip(1), block)
        if case["err"] > 0:
            hit = torch.rand((m, L), generator=gen, device="cuda") < case["err"]
            shift = torch.randint(1, 4, (m, L), generator=gen, device="cuda", dtype=torch.uint8)
            block = torch.where(hit, (block + shift) & 3, block)
        block = acgt[block.to(torch.int32)]
        parts.append(block[span < lengths[c:c + m, None]] if lo else block.reshape(-1))
    return torch.cat(parts), lengths


def _sets(case):
    """(reads, genome, k) of each read set of a case.  A batch holds six,
    log-spaced over a factor of 50, the largest with about half of the reads,
    k alternating with 21."""
    if case["kind"] != "batch":
        return [(case["reads"], case["genome"], case["k"])]
    w = [50.0 ** (-i / 5.0) for i in range(6)]
    n = [max(50, int(case["reads"] * x / sum(w))) for x in w]
    return [(n[i], int(case["genome"] * n[i] / case["reads"]) + 1000, case["k"] if i % 2 == 0 else 21)
            for i in range(6)]


# --------------------------------------------------------------------------
# room for the results
# --------------------------------------------------------------------------
def _shape(case, n, genome, k):
    """(bases, edge instances, k-mer positions, most distinct edges, most
    distinct nodes, most unitigs) of n reads.  The last three are what a
    program would size its buffers with: true (k+1)-mers number at most the
    genome's, and errors add at most one for each window that holds one
    (eight standard deviations on top), never more than the positions."""
    L, lo = case["read_len"], case["min_len"] or case["read_len"]
    span = L - lo + 1
    slack = 8.0 * L * math.sqrt(n) if span > 1 else 0.0
    N = n * sum(max(0, x - k) for x in range(lo, L + 1)) / span
    P = n * sum(max(0, x - k + 1) for x in range(lo, L + 1)) / span
    bases = n * (lo + L) / 2.0
    errors = bases * case["err"] + 8.0 * math.sqrt(bases * case["err"]) + 16
    wrong = lambda pos, m: pos * (1.0 - (1.0 - case["err"]) ** m) + 8.0 * m * math.sqrt(errors) if case["err"] else 0.0
    E = int(min(N + slack, genome + wrong(N, k + 1))) + 64
    V = int(min(P + slack, genome + wrong(P, k))) + 64
    # unitigs: islands of reads, at most four for each error, chance and repeat overlaps
    U = (min(n, 3.0 * n * math.exp(-N / genome) + 1000) + 4.0 * errors + 16.0 * V * V / 4.0 ** k
         + 0.1 * (case["repeats"] + case["tandem"]) * genome + 5000)
    return bases, N, P, E, V, int(min(U, V))


def _graph_room(E, V, W, **kw):
    size = {"V": V, "V1": V + 1, "E": E, "E2": 2 * E}
    return {f: torch.zeros(size[n] * (W if keyed else 1), dtype=ty, **kw) for f, n, ty, keyed in GRAPH_FIELDS}


def _unitig_room(V, U, k, **kw):
    return {"node_off": torch.zeros(U + 1, dtype=torch.int64, **kw), "nodes": torch.zeros(V, dtype=torch.int64, **kw),
            "seq_off": torch.zeros(U + 1, dtype=torch.int64, **kw),
            "seq": torch.zeros(V + U * (k - 1), dtype=torch.uint8, **kw),
            "circular": torch.zeros(U, dtype=torch.uint8, **kw)}


# --------------------------------------------------------------------------
# one pass
# --------------------------------------------------------------------------
def _start_reading(g, room):
    """Starts the copies of the graph's arrays into the program's buffers."""
    if (dbg.dbg_graph_num_edges(g) > room["src"].numel()
            or dbg.dbg_graph_num_nodes(g) >= room["row_ptr"].numel()):
        raise RuntimeError("the graph is larger than its buffers")
    o = {f: t.data_ptr() for f, t in room.items()}
    dbg.dbg_graph_nodes_async(g, keys=o["node_keys"])
    dbg.dbg_graph_edges_async(g, keys=o["edge_keys"], src=o["src"], dst=o["dst"], orient=o["orient"], mult=o["mult"])
    dbg.dbg_graph_csr_async(g, row_ptr=o["row_ptr"], nbr=o["adj_nbr"], edge=o["adj_edge"], role=o["adj_role"])


def _read_unitigs(u, room):
    if dbg.dbg_unitigs_count(u) > room["circular"].numel() or dbg.dbg_unitigs_total_bases(u) > room["seq"].numel():
        raise RuntimeError("the unitigs are larger than their buffers")
    dbg.dbg_unitigs_get_into(u, **{f: t.data_ptr() for f, t in room.items()})


def _put(room, got):
    """Host arrays into the program's own, by name."""
    for f, x in got.items():
        room[f][:len(x)] = x


def prepare(case, seed):
    kind, k = case["kind"], case["k"]
    ctx = dbg.Context()
    if case["tuned"]:
        dbg.dbg_autotune(ctx)
    st = {"kind": kind, "k": k, "ctx": ctx}
    if kind == "batch":
        st["sets"], st["room"] = [], []
        for i, (n, genome, kk) in enumerate(_sets(case)):
            r, l = _reads(case, n, genome, seed * 16 + i)
            st["sets"].append((r, l, kk))
            _, _, _, E, V, _ = _shape(case, n, genome, kk)
            st["room"].append(_graph_room(E, V, 1 if kk <= 31 else 2, device="cuda"))
        torch.cuda.synchronize()
        return st
    reads, lengths = _reads(case, case["reads"], case["genome"], seed)
    _, _, _, E, V, U = _shape(case, case["reads"], case["genome"], k)
    W = 1 if k <= 31 else 2
    torch.cuda.synchronize()
    if kind in ("compact", "simplify"):
        st["graph"] = dbg.dbg_build(ctx, reads, lengths, k)
        if kind == "compact":
            st["uroom"] = _unitig_room(V, U, k, device="cuda")
        else:
            st["room"] = {f: np.zeros(n, dtype=ty) for f, n, ty in
                          (("node_off", V + 1, np.uint64), ("nodes", V, np.uint64), ("seq_off", V + 1, np.uint64),
                           ("seq", V * k, np.uint8), ("circular", V, np.uint8), ("unit_a", E, np.uint32),
                           ("side_a", E, np.uint8), ("unit_b", E, np.uint32), ("side_b", E, np.uint8),
                           ("edge", E, np.uint32))}
        return st
    if kind == "counts":
        dbg.dbg_node_mult_set(ctx, True)
        dbg.dbg_node_reads_set(ctx, True)
        st["counts"] = {f: np.zeros(V, dtype=np.uint32) for f in ("node_mult", "node_reads", "roadmap")}
    if kind == "host":
        reads, lengths = reads.cpu().pin_memory(), lengths.cpu().numpy().view(np.uint32)
        st["room"], st["uroom"] = _graph_room(E, V, W, pin_memory=True), _unitig_room(V, U, k, pin_memory=True)
    else:
        st["room"] = _graph_room(E, V, W, device="cuda")
        if kind == "build_compact":
            st["uroom"] = _unitig_room(V, U, k, device="cuda")
    st["reads"], st["lengths"], st["budget"] = reads, lengths, case["budget_mb"] << 20
    torch.cuda.synchronize()
    return st


def _ints(room):
    """Host arrays as signed integers of the same bytes (torch has no arithmetic on unsigned ones)."""
    return {f: v.view(v.dtype.str.replace("u", "i")) if v.itemsize > 1 else v for f, v in room.items()}


def run(st):
    kind, k, ctx = st["kind"], st["k"], st["ctx"]
    if kind == "batch":
        graphs = dbg.dbg_build_batch(ctx, st["sets"])
        for g, room in zip(graphs, st["room"]):
            _start_reading(g, room)
        for g in graphs:
            dbg.dbg_graph_wait(g)
        return st["room"]
    if kind == "compact":
        _read_unitigs(dbg.dbg_compact(ctx, st["graph"]), st["uroom"])
        return st["uroom"]
    if kind == "simplify":
        got = dbg.dbg_simple_get(dbg.dbg_simplify(ctx, st["graph"], 3))
        removed = got.pop("removed")
        got["seq"] = np.frombuffer(got["seq"], dtype=np.uint8)
        _put(st["room"], got)
        return {"simple": _ints(st["room"]), "removed": removed}
    if kind == "bucketed":
        g = dbg.dbg_build_bucketed(ctx, st["reads"], st["lengths"], k, st["budget"])
    else:
        g = dbg.dbg_build(ctx, st["reads"], st["lengths"], k)
    _start_reading(g, st["room"])
    if kind == "host":  # the read-back overlaps the compaction
        _read_unitigs(dbg.dbg_compact(ctx, g), st["uroom"])
    dbg.dbg_graph_wait(g)
    if kind == "counts":
        _put(st["counts"], {"node_mult": dbg.dbg_graph_node_mult(g), "node_reads": dbg.dbg_graph_node_reads(g),
                            "roadmap": dbg.dbg_roadmap_nodes(ctx, g, 2)})
        return {"graph": st["room"], "counts": _ints(st["counts"])}
    if kind == "build_compact":
        _read_unitigs(dbg.dbg_compact(ctx, g), st["uroom"])
    return {"graph": st["room"], "unitigs": st["uroom"]} if "uroom" in st else st["room"]


# --------------------------------------------------------------------------
# the bytes a pass cannot do without
# --------------------------------------------------------------------------
def work(case):
    """Reads and lengths in, the result's arrays out, each once, at the sizes
    expected on average (|V| taken equal to |E|, unitigs counted by their
    nodes)."""
    kind = case["kind"]
    total = 0.0
    for n, genome, k in _sets(case):
        bases, N, _, E, _, _ = _shape(case, n, genome, k)
        seen = genome * (1.0 - math.exp(-N / genome))
        E = max(1.0, min(N, E, seen + N * (1.0 - (1.0 - case["err"]) ** (k + 1))))
        w = 8 if k <= 31 else 16
        graph = E * (2 * w + 8 + 13 + 18)
        chains = E * (8 + 2)
        if kind == "compact":
            total += E * (w + 8 + 18 + 1) + chains
        elif kind == "simplify":
            total += E * (w + 8 + 18 + 9) + chains + E
        else:
            total += bases + 4 * n + graph
            if kind in ("build_compact", "host"):
                total += chains
            if kind == "counts":
                total += 12 * E
    return {"bytes": total, "flops": 0.0}


def exact(case, seed):
    """Whole numbers only: they are equal or wrong."""
    return None
