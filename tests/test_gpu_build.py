"""The device CSR builder against a numpy sort: rows of every length class (a few entries up to rows too long
for a block's shared memory), one and two levels of splitting, repeated edges in each class, and
the core-ordered copy built from the same edges."""

import numpy as np
import pytest
import torch

import oracle
from paper_2606_07148_gb300 import ABCore, ABCoreError, abi

pytestmark = pytest.mark.gpu


def _rows(lengths, nV, rng):
    eu = np.repeat(np.arange(len(lengths)), lengths)
    ev = np.concatenate([rng.choice(nV, k, replace=False) for k in lengths])
    return eu, ev


def _random(nU, nV, m, rng):
    key = np.unique(rng.integers(0, nU * nV, m + m // 8 + 64))
    key = rng.permutation(key)[:m]
    return key // nV, key % nV


LENGTHS = [1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 257, 511, 513, 1000, 1023, 1024, 1025,
           1500, 2047, 2048, 2049, 3000, 4095, 4096, 4097, 5000, 8191, 8192, 8193, 12000]


def _graph(name):
    rng = np.random.default_rng(len(name))
    if name == "one":
        return 3, 2, *(np.array([x]) for x in (1, 1))
    if name == "bin-edges":      # rows that end where a bin ends, and bins that one row fills
        return _sized([4096, 4096, 2048, 2048, 1, 4095, 4097, 8192, 8191], 9000, rng)
    if name == "classes":        # every length class on the upper layer, single level
        return _sized(LENGTHS, 13000, rng)
    if name == "classes-lower":  # ... and on the lower one
        nV, nU, ev, eu = _sized(LENGTHS, 13000, rng)
        return nU, nV, eu, ev
    if name == "long":           # rows beyond shared memory, few of the edges
        nU, nV, eu, ev = _sized([30000, 26000, 24576, 20481, 20480] + LENGTHS, 31000, rng)
        fu, fv = _random(200000, 31000, 900000, rng)
        return nU + 200000, nV, np.concatenate([eu, fu + nU]), np.concatenate([ev, fv])
    if name == "long-whole":     # most edges in such rows: the layer is sorted whole
        return _sized([30000, 29000, 100, 5], 31000, rng)
    if name == "stars":          # one such row on each layer
        eu = np.concatenate([np.zeros(30000, np.int64), np.arange(1, 30000)])
        ev = np.concatenate([np.arange(30000), np.full(29999, 30000)])
        return 30000, 30001, eu, ev
    if name == "two-level":
        return 300007, 90001, *_random(300007, 90001, 4_700_000, rng)
    if name == "two-level-long":
        nU, nV, eu, ev = _sized([60000, 30000, 26000, 21000] + LENGTHS, 70000, rng)
        fu, fv = _random(400000, 70000, 5_000_000, rng)
        return nU + 400000, nV, np.concatenate([eu, fu + nU]), np.concatenate([ev, fv])
    if name == "two-level-whole":
        return _sized([26000] * 190, 30000, rng)
    raise ValueError(name)


def _sized(lengths, nV, rng):
    eu, ev = _rows(lengths, nV, rng)
    return len(lengths) + 2, nV, eu, ev


def _reference(nU, nV, eu, ev):
    du, dv = np.bincount(eu, minlength=nU), np.bincount(ev, minlength=nV)
    ou, ov = np.argsort(-du, kind="stable"), np.argsort(-dv, kind="stable")
    nu, nv = np.empty(nU, np.int64), np.empty(nV, np.int64)
    nu[ou], nv[ov] = np.arange(nU), np.arange(nV)
    x, y = nu[eu], nv[ev]
    a = np.lexsort((y, x))
    b = np.lexsort((x, y))
    off = np.concatenate([[0], np.cumsum(np.concatenate([du[ou], dv[ov]]))])
    return off, np.concatenate([y[a] + nU, x[b]]), np.concatenate([ou, ov])


NAMES = ["one", "bin-edges", "classes", "classes-lower", "long", "long-whole", "stars", "two-level", "two-level-long", "two-level-whole"]


@pytest.mark.parametrize("name", NAMES)
def test_rows_equal_a_sort(name):
    nU, nV, eu, ev = _graph(name)
    p = np.random.default_rng(1).permutation(len(eu))
    eu, ev = eu[p].astype(np.int32), ev[p].astype(np.int32)
    core = ABCore(0)
    core.load_edges(nU, nV, torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda())
    off, adj, n2o = core.export_csr()
    woff, wadj, wn2o = _reference(nU, nV, eu, ev)
    assert np.array_equal(off, woff) and np.array_equal(n2o, wn2o)
    assert np.array_equal(adj, wadj)
    core.close()


@pytest.mark.parametrize("length", [2, 5, 30, 33, 700, 1025, 4000, 9000, 26000])
def test_a_repeated_edge_is_refused(length):
    rng = np.random.default_rng(length)
    eu, ev = _rows([40, length, 3], 31000, rng)
    at = int(np.nonzero(eu == 1)[0][length // 2])
    eu, ev = np.append(eu, eu[at]).astype(np.int32), np.append(ev, ev[at]).astype(np.int32)
    core = ABCore(0)
    with pytest.raises(ABCoreError) as err:
        core.load_edges(4, 31000, torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda())
    assert err.value.code == abi.ABCORE_EEXIST
    core.load_edges(4, 31000, torch.from_numpy(eu[:-1]).cuda(), torch.from_numpy(ev[:-1]).cuda())
    core.close()


@pytest.mark.parametrize("name", ["classes", "long", "two-level"])
def test_core_ordered_copy(name):
    nU, nV, eu, ev = _graph(name)
    eu, ev = eu.astype(np.int32), ev.astype(np.int32)
    off, adj = oracle.build_csr(nU, nV, eu, ev)
    core = ABCore(0)
    core.load_edges(nU, nV, torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda())
    cu, cv, _ = core.core_numbers()
    want = oracle.core_numbers(nU, nV, off, adj)
    assert np.array_equal(np.concatenate([cu.cpu().numpy(), cv.cpu().numpy()]), want)
    core.set_param("algo", 2)
    for a, b in [(2, 5), (7, 3), (4, 40)]:
        wu, wv = oracle.peel(nU, nV, off, adj, a, b)
        mu, mv = core.compute(a, b)
        assert np.array_equal(mu.cpu().numpy(), wu) and np.array_equal(mv.cpu().numpy(), wv)
    core.close()
