"""The rules that pick the single peel's form by query: whatever they pick, and whatever a caller sets instead,
the masks are the oracle's. Counts in vertex order for some queries and spread for others, the first
round walked or queued, small and large grabs, pruned queries that leave nothing to peel, and a graph
large enough that the rule itself has the long first rounds walked without returns."""

import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2606_07148_gb300 import ABCore

pytestmark = pytest.mark.gpu

NU, NV, M = 300_001, 150_003, 12_000_000


@pytest.fixture(scope="module")
def graph():
    eu, ev = synth.chung_lu_edges(NU, NV, M, 2.1, 2.4, 3, device="cuda")
    off, adj = oracle.build_csr(NU, NV, eu.cpu().numpy(), ev.cpu().numpy())
    core = ABCore(0)
    core.load_edges(NU, NV, eu, ev)
    yield eu, ev, off, adj, core
    core.close()


PAIRS = [(1, 1), (2, 2), (12, 30), (40, 40), (60, 60), (90, 20), (30, 150), (400, 400)]


def test_every_form_gives_the_same_cores(graph):
    eu, ev, off, adj, core = graph
    want = {p: oracle.peel(NU, NV, off, adj, *p) for p in PAIRS}
    for setting in ({}, {"round0": 0}, {"round0": 1, "round0_variant": 4}, {"round0": 0, "count_swizzle": 0}, {"grab_div": 1}, {"grab_div": 1 << 20},
                    {"flush_steps": 1, "mode": 0}, {"mode": 3, "emit_scatter_max_pct": 100}, {"mode": 1, "emit_scatter_max_pct": 0}):
        c = core
        if setting:
            c = ABCore(0)
            c.load_edges(NU, NV, eu, ev)
            for k, v in setting.items():
                c.set_param(k, v)
        for p in PAIRS:
            mu, mv = c.compute(*p)
            assert np.array_equal(mu.cpu().numpy(), want[p][0]) and np.array_equal(mv.cpu().numpy(), want[p][1]), (setting, p)
        if setting:
            c.close()


@pytest.mark.parametrize("scatter_pct", [0, 5, 100])
def test_pruned_queries_with_nothing_to_peel(graph, scatter_pct):
    eu, ev, off, adj, core = graph
    c = ABCore(0)
    c.load_edges(NU, NV, eu, ev)
    _, _, top = c.core_numbers()
    c.set_param("algo", 2)
    c.set_param("emit_scatter_max_pct", scatter_pct)
    for a, b in [(0, 0), (1, 1), (2, 2), (top // 2, top // 2), (top, top), (top + 1, top + 1), (5, 9), (10_000, 3)]:
        wu, wv = oracle.peel(NU, NV, off, adj, a, b)
        for shift in (0, 1):
            mu = torch.full((NU + shift,), 5, dtype=torch.uint8, device="cuda")[shift:]
            mv = torch.full((NV + shift,), 5, dtype=torch.uint8, device="cuda")[shift:]
            c.compute(a, b, mu, mv, asynchronous=True)
            c.compute(4, 7)  # (a peel right after it finds its bitmap and queue as it left them)
            c.sync()
            assert np.array_equal(mu.cpu().numpy(), wu) and np.array_equal(mv.cpu().numpy(), wv), (a, b, shift)
    c.close()


def test_long_first_rounds_are_walked():
    nU, nV, eu, ev = synth.make_graph("peel-4Mx2M-80M", device="cuda")
    off, adj = oracle.build_csr(nU, nV, eu.cpu().numpy(), ev.cpu().numpy())
    core = ABCore(0)
    core.load_edges(nU, nV, eu, ev)
    pairs = [(50, 50), (20, 100), (2, 2)]
    want = oracle.peel_many(nU, nV, off, adj, pairs)
    for a, b in pairs:
        wu, wv, _ = want[a, b]
        core.set_param("reset_stats", 1)
        mu, mv = core.compute(a, b)
        assert np.array_equal(mu.cpu().numpy(), wu) and np.array_equal(mv.cpu().numpy(), wv), (a, b)
        assert (core.stats()["round0_rows"] > 0) == (a > 2), (a, b)
    core.close()


def test_a_chosen_form_is_used_where_the_rule_walks():
    nU, nV, eu, ev = synth.make_graph("peel-4Mx2M-80M", device="cuda")
    off, adj = oracle.build_csr(nU, nV, eu.cpu().numpy(), ev.cpu().numpy())
    wu, wv, _ = oracle.peel_many(nU, nV, off, adj, [(50, 50)])[50, 50]
    core = ABCore(0)
    core.load_edges(nU, nV, eu, ev)
    for variant in (None, 5, 0, 2):  # (None: by rule, rows without the hub table at this length)
        if variant is not None:
            core.set_param("round0_variant", variant)
        core.set_param("reset_stats", 1)
        mu, mv = core.compute(50, 50)
        assert np.array_equal(mu.cpu().numpy(), wu) and np.array_equal(mv.cpu().numpy(), wv), variant
        st = core.stats()
        assert st["round0_rows"] > 0 and (st["hub_decrements"] > 0) == (variant == 5), variant
    core.close()


@pytest.mark.parametrize("pair", [(200, 200), (200, 201), (256, 20), (257, 20), (20, 257), (500, 500)])
def test_large_bounds(pair):
    # at and past the bounds from which first rounds are queued and pushes handed over at once
    nU, nV = 20001, 10003
    eu, ev = synth.chung_lu_edges(nU, nV, 3_000_000, 2.1, 2.2, 5, device="cuda")
    off, adj = oracle.build_csr(nU, nV, eu.cpu().numpy(), ev.cpu().numpy())
    wu, wv, _ = oracle.peel_many(nU, nV, off, adj, [pair])[pair]
    core = ABCore(0)
    core.load_edges(nU, nV, eu, ev)
    for setting in ({}, {"round0": 1}, {"flush_steps": 16}):
        for k, v in setting.items():
            core.set_param(k, v)
        mu, mv = core.compute(*pair)
        assert np.array_equal(mu.cpu().numpy(), wu) and np.array_equal(mv.cpu().numpy(), wv), setting
    core.close()
