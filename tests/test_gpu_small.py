"""The one-block peel of small graphs against the oracle and the general peel: layer sizes with and without
four-id mask words, bounds of zero, cores that keep everything and nothing, long cascades, the pruned
query, batches up to the largest graph one block holds, and the edge of the rule that picks it."""

import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2606_07148_gb300 import ABCore

pytestmark = pytest.mark.gpu


def _chain(n):
    # u0 v0 u1 v1 ...: peeling (2, 2) removes it vertex by vertex from both ends
    e = [(i, i) for i in range(n)] + [(i + 1, i) for i in range(n - 1)]
    return n, n, np.array(e, dtype=np.int32)


def _graph(name):
    if name == "chain":
        nU, nV, e = _chain(600)
        return nU, nV, e[:, 0].copy(), e[:, 1].copy()
    if name == "empty":
        return 7, 5, np.zeros(0, np.int32), np.zeros(0, np.int32)
    nU, nV, m = {"even": (2000, 1500, 20000), "odd": (2001, 1499, 20000), "tiny": (5, 3, 11), "most": (9001, 7383, 120000)}[name]
    eu, ev = synth.chung_lu_edges(nU, nV, m, 2.2, 2.3, 5)
    return nU, nV, eu.numpy(), ev.numpy()


PAIRS = [(0, 0), (0, 3), (4, 0), (1, 1), (2, 2), (2, 3), (5, 5), (9, 4), (30, 30), (1000, 1), (1, 100000)]


@pytest.mark.parametrize("name", ["even", "odd", "tiny", "chain", "empty", "most"])
def test_queries_and_batch_equal_the_oracle(name):
    nU, nV, eu, ev = _graph(name)
    off, adj = oracle.build_csr(nU, nV, eu, ev)
    want = [oracle.peel(nU, nV, off, adj, a, b) for a, b in PAIRS]
    core = ABCore(0)
    core.load_edges(nU, nV, torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda())
    for small in (1, 0):
        core.set_param("small_peel", small)
        for shift in (0, 1):  # (masks at odd addresses take the byte stores)
            du = torch.full((len(PAIRS) * nU + shift,), 9, dtype=torch.uint8, device="cuda")[shift:].view(len(PAIRS), nU)
            dv = torch.full((len(PAIRS) * nV + shift,), 9, dtype=torch.uint8, device="cuda")[shift:].view(len(PAIRS), nV)
            core.compute_batch([p[0] for p in PAIRS], [p[1] for p in PAIRS], du, dv)
            qs = [core.compute(a, b, torch.full((nU + shift,), 9, dtype=torch.uint8, device="cuda")[shift:],
                               torch.full((nV + shift,), 9, dtype=torch.uint8, device="cuda")[shift:], asynchronous=True) for a, b in PAIRS]
            core.sync()
            for k, (wu, wv) in enumerate(want):
                assert np.array_equal(du[k].cpu().numpy(), wu) and np.array_equal(dv[k].cpu().numpy(), wv), (small, PAIRS[k])
                assert np.array_equal(qs[k][0].cpu().numpy(), wu) and np.array_equal(qs[k][1].cpu().numpy(), wv), (small, PAIRS[k])
    if name != "empty":
        core.core_numbers()
        core.set_param("algo", 2)
        core.set_param("small_peel", 1)
        for k, (a, b) in enumerate(PAIRS):
            mu, mv = core.compute(a, b)
            assert np.array_equal(mu.cpu().numpy(), want[k][0]) and np.array_equal(mv.cpu().numpy(), want[k][1]), ("pruned", a, b)
    core.close()


@pytest.mark.parametrize("nU,nV", [(20000, 16000), (20001, 16000), (9000, 7384), (9000, 7385)])
def test_sizes_at_the_limits(nU, nV):
    # 36,000 vertices: the last batch a block per pair takes; 16,384: the last query one block takes
    eu, ev = synth.chung_lu_edges(nU, nV, 12 * nU, 2.2, 2.3, 9)
    off, adj = oracle.build_csr(nU, nV, eu.numpy(), ev.numpy())
    core = ABCore(0)
    core.load_edges(nU, nV, eu.cuda(), ev.cuda())
    pairs = [(1, 1), (0, 0), (3, 4), (8, 8)]
    bu, bv = core.compute_batch([p[0] for p in pairs], [p[1] for p in pairs])
    for k, (a, b) in enumerate(pairs):
        wu, wv = oracle.peel(nU, nV, off, adj, a, b)
        mu, mv = core.compute(a, b)
        assert np.array_equal(bu[k].cpu().numpy(), wu) and np.array_equal(bv[k].cpu().numpy(), wv)
        assert np.array_equal(mu.cpu().numpy(), wu) and np.array_equal(mv.cpu().numpy(), wv)
    core.close()


def test_contexts_of_different_sizes_in_turn():
    # each launch's shared-memory need differs; the limit set for one context must not bind another
    graphs = [_graph(n) for n in ("tiny", "most", "even")]
    cores = []
    for nU, nV, eu, ev in graphs:
        c = ABCore(0)
        c.load_edges(nU, nV, torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda())
        cores.append((c, oracle.build_csr(nU, nV, eu, ev)))
    for _ in range(2):
        for (c, (off, adj)), (nU, nV, _, _) in zip(cores, graphs):
            wu, wv = oracle.peel(nU, nV, off, adj, 2, 2)
            mu, mv = c.compute(2, 2)
            bu, bv = c.compute_batch([2], [2])
            assert np.array_equal(mu.cpu().numpy(), wu) and np.array_equal(mv.cpu().numpy(), wv)
            assert np.array_equal(bu[0].cpu().numpy(), wu) and np.array_equal(bv[0].cpu().numpy(), wv)
    for c, _ in cores:
        c.close()
