"""Core numbers where long rows matter: rows whose values do not fit in shared memory, in one step of counts and in several,
rows around the sizes at which the search for their end changes, and hubs among an ordinary graph."""

import time

import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2606_07148_gb300 import ABCore

pytestmark = pytest.mark.gpu


def _with_hubs(k, per, nU, nV, m, seed):
    """An ordinary graph and k upper vertices with `per` random lower neighbours each."""
    eu, ev = synth.chung_lu_edges(nU, nV, m, 2.1, 2.3, seed)
    rng = np.random.default_rng(seed)
    hu = np.repeat(np.arange(k, dtype=np.int32), per) + nU
    hv = np.concatenate([rng.permutation(nV)[:per].astype(np.int32) for _ in range(k)])
    return nU + k, nV, np.concatenate([eu.numpy(), hu]), np.concatenate([ev.numpy(), hv])


def _check(nU, nV, eu, ev):
    off, adj = oracle.build_csr(nU, nV, eu, ev)
    want = oracle.core_numbers(nU, nV, off, adj)
    core = ABCore(0)
    core.load_edges(nU, nV, torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda())
    cu, cv, mx = core.core_numbers()
    got = np.concatenate([cu.cpu().numpy(), cv.cpu().numpy()])
    assert np.array_equal(got, want) and mx == want.max()
    core.close()


@pytest.mark.parametrize("per", [513, 514, 769, 4095, 4096, 4097, 20_000, 32_768, 32_769, 36_865, 66_000])
def test_hubs_among_an_ordinary_graph(per):
    _check(*_with_hubs(7, per, 40_000, 70_000, 900_000, per))


@pytest.mark.parametrize("more", [0, 30_000])
def test_a_row_whose_value_falls_by_thousands(more):
    # a hub whose 4,600 neighbours have 4,400 others each, all of low degree: its first value is 4,401, its core number 2
    # (with 30,000 more of degree 1 its row is one of those the whole grid takes)
    hubs, leaves = 4600, 4400
    pool = hubs * leaves // 2
    k = np.random.default_rng(1).permutation(hubs * leaves)
    lu, lv = (k % pool).astype(np.int32), (k // leaves).astype(np.int32)  # (a leaf twice at most, at different hubs)
    nU, nV = pool + 1, hubs + more
    _check(nU, nV, np.concatenate([lu, np.full(nV, pool, np.int32)]), np.concatenate([lv, np.arange(nV, dtype=np.int32)]))


@pytest.mark.parametrize("k", [255, 256, 257, 300])
def test_more_rows_of_the_grid_than_a_batch(k):
    # k rows of 33,000 or so in one layer, some of them neighbours of two such rows in the other
    rng = np.random.default_rng(k)
    nV = 34_000
    u = np.repeat(np.arange(k, dtype=np.int32), nV)
    v = np.tile(np.arange(nV, dtype=np.int32), k)
    keep = rng.random(len(u)) < 0.975
    extra = np.arange(40_000, dtype=np.int32) + k  # the upper layer's other vertices: two lower hubs reach them
    eu = np.concatenate([u[keep], extra, extra])
    ev = np.concatenate([v[keep], np.full(40_000, 5, np.int32), np.full(40_000, 7, np.int32)])
    _check(k + 40_000, nV, eu, ev)


def test_hubs_take_no_longer_than_building_the_graph_does():
    # (20 rows of 400,000: 99 % of it was the search for their values)
    nU, nV, eu, ev = _with_hubs(20, 400_000, 800_000, 400_000, 8_000_000, 3)
    core = ABCore(0)
    eu, ev = torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda()
    load, cores = [], []
    for _ in range(4):
        torch.cuda.synchronize()
        t = time.perf_counter()
        core.load_edges(nU, nV, eu, ev)
        load.append(time.perf_counter() - t)
        t = time.perf_counter()
        core.core_numbers()
        cores.append(time.perf_counter() - t)
    core.close()
    assert min(cores) < 4 * min(load), (load, cores)
