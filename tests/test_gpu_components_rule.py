"""Labels on both sides of the rule that unites a sparse graph's edges in one launch: around 131,072 edges and two edges a
vertex, chains, stars and many small components, equal to the oracle's, communities and updates among them."""

import numpy as np
import pytest
import torch

import oracle
from paper_2606_07148_gb300 import ABCore, abi

pytestmark = pytest.mark.gpu


def _graph(shape, m, rng):
    if shape == "path":
        i = np.arange(m + 1)
        return m // 2 + 1, m // 2 + 1, (i[:-1] + 1) // 2, i[:-1] // 2
    if shape == "stars":  # one lower hub a star, which shares a leaf with the next
        i = np.arange(m)
        return m, m // 1500 + 2, i - i // 1500, i // 1500
    if shape == "bicliques":
        i = np.arange(m // 4 * 4)
        return m // 2 + 5, m // 2 + 7, i // 4 * 2 + i % 4 // 2, i // 4 * 2 + i % 2
    # "two": exactly two edges a vertex or just more, random
    n = m // 4
    key = np.unique(rng.integers(0, n * n, m + m // 50))
    key = rng.permutation(key)[:m]
    return n, n, key // n, key % n


@pytest.mark.parametrize("shape", ["path", "stars", "bicliques", "two"])
@pytest.mark.parametrize("m", [40, 6000, (1 << 17) - 1, 1 << 17, (1 << 17) + 1, 140_000])
def test_labels_and_launches(shape, m):
    rng = np.random.default_rng(m)
    nU, nV, eu, ev = _graph(shape, m, rng)
    p = rng.permutation(len(eu))
    pu, pv = rng.permutation(nU).astype(np.int32), rng.permutation(nV).astype(np.int32)
    eu, ev = pu[eu[p]], pv[ev[p]]
    off, adj = oracle.build_csr(nU, nV, eu, ev)
    want, wn = oracle.components(nU, nV, off, adj)
    core = ABCore(0)
    core.load_edges(nU, nV, torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda())
    core.components()
    core.set_param("reset_stats", 1)
    lu, lv, nc = core.components()
    launches = core.stats()["launches"]
    assert nc == wn and np.array_equal(np.concatenate([lu.cpu().numpy(), lv.cpu().numpy()]), want)
    linked = len(np.unique(eu)) + len(np.unique(ev))
    whole = len(eu) <= 1 << 17 and len(eu) <= 2 * linked
    assert (launches <= 4) == whole, launches  # (a forest, its edges, the roots' names, the labels)
    q = int(eu[0])
    gu, gv, size = core.community(0, q, 1, 1)
    got = np.concatenate([gu.cpu().numpy(), gv.cpu().numpy()]).astype(bool)
    assert size == int(got.sum()) and np.array_equal(got, want == want[q])
    core.close()


def test_updates_of_a_sparse_graph():
    # the forest under deletes and inserts (tombstones, a kept component), in the served and the component-scoped form
    rng = np.random.default_rng(5)
    nU, nV, eu, ev = _graph("path", 3000, rng)
    eu, ev = eu.astype(np.int32), ev.astype(np.int32)
    for scope in (0, 1):
        core = ABCore(0)
        core.set_param("query_scope", scope)
        core.load_edges(nU, nV, torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda())
        cur = set(zip(eu.tolist(), ev.tolist()))
        for k in (5, 1500, 2999, 700):
            core.query_edge(int(eu[k]), int(ev[k]), abi.ABCORE_DELETE, 1, 1)
            cur.discard((int(eu[k]), int(ev[k])))
        core.query_edge(3, nV - 1, abi.ABCORE_INSERT, 1, 1)
        cur.add((3, nV - 1))
        e = np.array(sorted(cur), dtype=np.int32)
        off, adj = oracle.build_csr(nU, nV, np.ascontiguousarray(e[:, 0]), np.ascontiguousarray(e[:, 1]))
        want, wn = oracle.components(nU, nV, off, adj)
        lu, lv, nc = core.components()
        assert nc == wn and np.array_equal(np.concatenate([lu.cpu().numpy(), lv.cpu().numpy()]), want), scope
        core.close()
