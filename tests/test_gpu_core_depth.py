"""Core numbers of deep graphs: paths, cycles with tails, grids, trees and combs, whose values settle over as many rounds as they
are deep; equal to the oracle's, whatever the limit of the device waits, and no slower than a peel of the same graph."""

import time

import numpy as np
import pytest
import torch

import oracle
from paper_2606_07148_gb300 import ABCore

pytestmark = pytest.mark.gpu


def _bipartite(n, a, b, colour, rng):
    """Edges (a, b) over vertices 0..n-1 of two colours as a graph with random ids in each layer."""
    ident = np.empty(n, dtype=np.int32)
    for c in (0, 1):
        k = np.flatnonzero(colour == c)
        ident[k] = rng.permutation(len(k))
    u, v = np.where(colour[a] == 0, a, b), np.where(colour[a] == 0, b, a)
    p = rng.permutation(len(a))
    return int((colour == 0).sum()), int((colour == 1).sum()), ident[u][p], ident[v][p]


def _path(n, rng):
    i = np.arange(n)
    return _bipartite(n, i[:-1], i[1:], i % 2, rng)


def _grid(w, h, rng):
    i = np.arange(w * h).reshape(w, h)
    a = np.concatenate([i[:-1].ravel(), i[:, :-1].ravel()])
    b = np.concatenate([i[1:].ravel(), i[:, 1:].ravel()])
    return _bipartite(w * h, a, b, (np.add.outer(np.arange(w), np.arange(h)) % 2).ravel(), rng)


def _comb(n, tooth, rng):
    """A cycle of n vertices, each with a path of `tooth` more, and a hub on one of them."""
    i = np.arange(n)
    a, b, col, last, total = [i], [(i + 1) % n], [i % 2], i, n
    for k in range(tooth):
        new = total + i
        a.append(last)
        b.append(new)
        col.append((i + k + 1) % 2)
        last, total = new, total + n
    hub = total + np.arange(700)
    a.append(np.zeros(700, dtype=np.int64))
    b.append(hub)
    col.append(np.ones(700, dtype=np.int64))
    return _bipartite(total + 700, np.concatenate(a), np.concatenate(b), np.concatenate(col), rng)


def _tree(depth, rng):
    i = np.arange(1, 2 ** depth - 1)
    level = np.floor(np.log2(np.arange(2 ** depth - 1) + 1)).astype(int)
    return _bipartite(2 ** depth - 1, (i - 1) // 2, i, level % 2, rng)


GRAPHS = {
    "path": lambda r: _path(30_001, r), "two": lambda r: _path(2, r), "grid": lambda r: _grid(90, 71, r), "strip": lambda r: _grid(3, 4000, r),
    "comb": lambda r: _comb(40, 300, r), "wide comb": lambda r: _comb(400, 20, r), "cycle with teeth": lambda r: _comb(1000, 1, r), "tree": lambda r: _tree(14, r),
}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("timeout", [4000, 5])
def test_core_numbers_equal_the_oracle(name, timeout):
    nU, nV, eu, ev = GRAPHS[name](np.random.default_rng(len(name)))
    off, adj = oracle.build_csr(nU, nV, eu, ev)
    want = oracle.core_numbers(nU, nV, off, adj)
    core = ABCore(0)
    core.set_param("timeout_ms", timeout)
    core.load_edges(nU, nV, torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda())
    cu, cv, mx = core.core_numbers()
    assert np.array_equal(np.concatenate([cu.cpu().numpy(), cv.cpu().numpy()]), want) and mx == want.max()
    core.close()


def test_a_path_takes_no_longer_than_its_peel():
    # the (2,2)-peel of a path removes it vertex by vertex from both ends, which is as deep as its core numbers are
    nU, nV, eu, ev = _path(100_001, np.random.default_rng(2))
    core = ABCore(0)
    core.set_param("algo", 1)
    core.load_edges(nU, nV, torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda())
    best = {"peel": 1e9, "cores": 1e9}
    core.compute(2, 2)
    for _ in range(3):
        torch.cuda.synchronize()
        t = time.perf_counter()
        core.compute(2, 2)
        torch.cuda.synchronize()
        best["peel"] = min(best["peel"], time.perf_counter() - t)
        core.load_edges(nU, nV, torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda())
        t = time.perf_counter()
        core.core_numbers()
        best["cores"] = min(best["cores"], time.perf_counter() - t)
    core.close()
    assert best["cores"] < 1.25 * best["peel"] + 0.002, best
