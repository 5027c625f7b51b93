"""Long rows in the one-block peel: they are walked by the whole block, up to 64 of them a level, the rest by eight lanes
each; graphs of few vertices with rows of thousands of entries, none slower in one block than in the general peel."""

import time

import numpy as np
import pytest
import torch

import oracle
from paper_2606_07148_gb300 import ABCore

pytestmark = pytest.mark.gpu


def _full(a, b, rng, drop):
    """a x b, all edges but `drop` random ones, in random order."""
    k = rng.permutation(a * b)[drop:]
    return a, b, (k // b).astype(np.int32), (k % b).astype(np.int32)


def _graphs():
    rng = np.random.default_rng(4)
    yield "few long rows", _full(16, 16000, rng, 1), [(16000, 16), (15999, 16), (16000, 15), (15990, 17)]
    yield "two long rows", _full(2, 16001, rng, 1), [(16001, 2), (16000, 2)]
    yield "more long rows than are listed", _full(100, 2500, rng, 1), [(2500, 100), (2499, 100), (1, 100), (2500, 1)]
    for w in (2047, 2048, 2049, 2303, 2304, 2305, 4097):
        yield "rows of %d" % w, _full(10, w, rng, 7), [(w, 10), (w - 1, 10), (w, 9), (3, 3)]
    # rows whose first entries alone are candidates: half of the lower layer has one edge less than its bound
    nU, nV, u, v = _full(9, 7000, rng, 0)
    keep = ~((u == 0) & (v % 2 == 0))
    yield "long rows of few candidates", (nU, nV, u[keep], v[keep]), [(5000, 9), (3500, 9), (7000, 8), (7000, 9)]


GRAPHS = list(_graphs())


@pytest.mark.parametrize("name,graph,pairs", GRAPHS, ids=[g[0].replace(" ", "-") for g in GRAPHS])
def test_cores_equal_the_oracle(name, graph, pairs):
    nU, nV, eu, ev = graph
    off, adj = oracle.build_csr(nU, nV, eu, ev)
    core = ABCore(0)
    core.load_edges(nU, nV, torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda())
    pairs = pairs + [(1, 1), (nV // 2, nU // 2)]
    want = [oracle.peel(nU, nV, off, adj, a, b) for a, b in pairs]
    for algo in (1, 2):  # (2: pruned by core numbers, some candidates are certain)
        core.set_param("algo", algo)
        bu, bv = core.compute_batch([p[0] for p in pairs], [p[1] for p in pairs])
        for k, (a, b) in enumerate(pairs):
            mu, mv = core.compute(a, b)
            assert np.array_equal(mu.cpu().numpy(), want[k][0]) and np.array_equal(mv.cpu().numpy(), want[k][1]), (algo, a, b)
            assert np.array_equal(bu[k].cpu().numpy(), want[k][0]) and np.array_equal(bv[k].cpu().numpy(), want[k][1]), (a, b)
    core.close()


def _hubs(k, w):
    """k hubs over w lower vertices; one lower vertex lacks hub 0, which has one of its own instead: all hubs fall at once
    for (w, k), and everything with them."""
    nU, nV, u, v = _full(k, w, np.random.default_rng(1), 0)
    v = np.where((u == 0) & (v == 0), w, v).astype(np.int32)
    return nU, nV + 1, u, v


@pytest.mark.parametrize("graph,pair", [(_full(16, 16000, np.random.default_rng(1), 1), (16000, 16)), (_full(2, 16000, np.random.default_rng(1), 1), (16000, 2)),
                                        (_hubs(30, 8000), (8000, 30)), (_hubs(3, 16000), (16000, 3))])
def test_no_slower_than_the_general_peel(graph, pair):
    nU, nV, eu, ev = graph
    off, adj = oracle.build_csr(nU, nV, eu, ev)
    wu, wv = oracle.peel(nU, nV, off, adj, *pair)
    core = ABCore(0)
    core.load_edges(nU, nV, torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda())
    mu, mv = core.compute(*pair)
    assert np.array_equal(mu.cpu().numpy(), wu) and np.array_equal(mv.cpu().numpy(), wv)
    best = {}
    for small in (1, 0):
        core.set_param("small_peel", small)
        for _ in range(30):
            torch.cuda.synchronize()
            t = time.perf_counter()
            core.compute(*pair, mu, mv)
            best[small] = min(best.get(small, 1.0), time.perf_counter() - t)
    core.close()
    assert best[1] < 1.25 * best[0], best  # (quickest of 30 each)
