"""A context's C handle goes after those of its results, whichever is closed
or collected first: results release their memory on the context's stream."""
from __future__ import annotations

import gc

import pytest

from paper_1003_1940_gb300 import dbg


class Fake:
    def __init__(self):
        self.calls = []

    def __getattr__(self, name):
        return lambda handle: self.calls.append((name, handle))


@pytest.fixture()
def lib(monkeypatch):
    gc.collect()  # (other tests' handles are the real library's)
    fake = Fake()
    monkeypatch.setattr(dbg, "_lib", fake)
    return fake


def context(handle):
    ctx = object.__new__(dbg.Context)
    ctx.handle = handle
    ctx._live, ctx._dying = set(), []
    return ctx


def test_context_closed_first(lib):
    ctx = context("c")
    g, u, s = dbg.Graph(ctx, "g"), dbg.Unitigs(ctx, "u"), dbg.Simple(ctx, "s")
    ctx.close()
    ctx.close()
    assert lib.calls == [] and ctx.handle is None
    u.free()
    g.free()
    g.free()
    assert lib.calls == [("dbg_unitigs_free", "u"), ("dbg_graph_free", "g")]
    del s
    assert lib.calls[2:] == [("dbg_simple_free", "s"), ("dbg_destroy", "c")]


def test_results_freed_first(lib):
    ctx = context("c")
    dbg.Graph(ctx, "g").free()
    ctx.close()
    assert lib.calls == [("dbg_graph_free", "g"), ("dbg_destroy", "c")]


@pytest.mark.parametrize("context_first", [True, False])
def test_collected_as_a_cycle(lib, context_first):
    """A program's globals at exit: one cycle with its functions."""
    box = {}
    ctx = context("c")
    if context_first:
        box["ctx"] = ctx
    box["graphs"] = [dbg.Graph(ctx, f"g{i}") for i in range(3)]
    box["ctx"] = ctx
    box["self"] = box
    del box, ctx
    gc.collect()
    assert sorted(lib.calls[:3]) == [("dbg_graph_free", f"g{i}") for i in range(3)]
    assert lib.calls[3:] == [("dbg_destroy", "c")]
