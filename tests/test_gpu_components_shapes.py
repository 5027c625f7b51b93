"""Component labels and communities on graphs whose shape decides which edges the sampled union-find
looks at: trees that the first-neighbour seed leaves apart, components that do not hold the first U
vertex, rows of every length class on both layers, and cores without the leading vertices."""

import numpy as np
import pytest
import torch

import oracle
from paper_2606_07148_gb300 import ABCore

pytestmark = pytest.mark.gpu


def _biclique(u0, v0, a, b):
    return [(u0 + i, v0 + j) for i in range(a) for j in range(b)]


def _graph(shape):
    rng = np.random.default_rng(11)
    if shape == "path":          # u0 v0 u1 v1 ...: long chains, every degree 1 or 2
        e = [(i, i) for i in range(700)] + [(i + 1, i) for i in range(699)]
        return 705, 703, e
    if shape == "stars":         # hub rows on both layers (>= 1024), joined by one edge at their ends
        e = [(0, j) for j in range(1500)] + [(i, 1500) for i in range(1, 1400)] + [(1399, 1499)]
        return 1500, 1600, e
    if shape == "equal":         # equal components: none holds more than its share
        e = sum((_biclique(40 * k, 33 * k, 40, 33) for k in range(30)), [])
        return 1203, 1001, e
    if shape == "chained":       # dense blocks that only low-degree vertices join
        e = sum((_biclique(50 * k, 50 * k, 45, 45) for k in range(12)), [])
        e += [(50 * k + 47, 50 * k) for k in range(12)] + [(50 * k + 47, 50 * (k + 1)) for k in range(11)]
        return 600, 600, e
    # sparse random: many components of all sizes and isolated vertices
    e = {(int(u), int(v)) for u, v in zip(rng.integers(0, 5000, 3500), rng.integers(0, 4000, 3500))}
    return 5000, 4000, sorted(e)


@pytest.mark.parametrize("shape", ["path", "stars", "equal", "chained", "sparse"])
def test_labels_and_communities(shape):
    nU, nV, edges = _graph(shape)
    e = np.array(edges, dtype=np.int32)[np.random.default_rng(3).permutation(len(edges))]
    eu, ev = np.ascontiguousarray(e[:, 0]), np.ascontiguousarray(e[:, 1])
    off, adj = oracle.build_csr(nU, nV, eu, ev)
    core = ABCore(0)
    core.load_edges(nU, nV, torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda())
    want, wn = oracle.components(nU, nV, off, adj)
    lu, lv, nc = core.components()
    assert nc == wn
    assert np.array_equal(np.concatenate([lu.cpu().numpy(), lv.cpu().numpy()]), want)
    for a, b in [(1, 1), (2, 2), (33, 40), (45, 45)]:
        mu, mv = (x.astype(bool) for x in oracle.peel(nU, nV, off, adj, a, b))
        live = mu[eu] & mv[ev]
        o2, a2 = oracle.build_csr(nU, nV, np.ascontiguousarray(eu[live]), np.ascontiguousarray(ev[live]))
        lab, _ = oracle.components(nU, nV, o2, a2)
        member = np.concatenate([mu, mv])
        for q in (0, nU // 2, int(np.argmax(mu)), nU - 1):
            w = member & (lab == lab[q]) & mu[q]
            gu, gv, size = core.community(0, q, a, b)
            got = np.concatenate([gu.cpu().numpy(), gv.cpu().numpy()]).astype(bool)
            assert size == int(w.sum()) and np.array_equal(got, w), (shape, a, b, q)
    core.close()
