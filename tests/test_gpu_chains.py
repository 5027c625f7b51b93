"""Batch chains and the general peel on graphs that the one-block kernels would take: a parameter of theirs that a caller
sets is followed, and the chains' own forms (32-bit counts, rows of steps of every width, more chains than a wave,
several waves, a captured plan replayed into other buffers) equal the oracle."""

import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2606_07148_gb300 import ABCore

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def small():
    nU, nV = 2000, 1500
    eu, ev = synth.chung_lu_edges(nU, nV, 20000, 2.2, 2.3, 5)
    off, adj = oracle.build_csr(nU, nV, eu.numpy(), ev.numpy())
    return nU, nV, eu, ev, off, adj


def _check(core, nU, nV, off, adj, pairs, chains):
    core.set_param("reset_stats", 1)
    mu, mv = core.compute_batch([p[0] for p in pairs], [p[1] for p in pairs])
    # the one-block kernel is one launch a batch; a wave of chains is two, the chains and their masks
    assert (core.stats()["launches"] > 1) == chains
    for k, (a, b) in enumerate(pairs):
        wu, wv = oracle.peel(nU, nV, off, adj, a, b)
        assert np.array_equal(mu[k].cpu().numpy(), wu) and np.array_equal(mv[k].cpu().numpy(), wv), (a, b)


KERNELS = [("chunk", 64), ("batch_entries", 256), ("flush_steps", 2), ("blocks_per_sm", 2), ("mode", 1), ("hub_degree", 64), ("probe_bytes", 12)]
PEEL = [("grab_div", 8), ("local_rounds", 4), ("batch_entries_small", 0), ("round0", 0), ("round0", 1), ("round0_variant", 4),
        ("round0_hub", 64), ("count_swizzle", 0), ("pdl", 0), ("emit_scatter_max_pct", 50), ("emit_bitmap_min_pct", 101)]
CHAINS = [("packed_counts", 0), ("batch_wave", 3), ("batch_seed", 1), ("batch_plain_below", 2)]


@pytest.mark.parametrize("name,value", [(None, 0)] + KERNELS + PEEL + CHAINS)
def test_a_set_parameter_is_followed(small, name, value):
    nU, nV, eu, ev, off, adj = small
    core = ABCore(0)
    core.load_edges(nU, nV, eu.cuda(), ev.cuda())
    if name:
        core.set_param(name, value)
    core.set_param("reset_stats", 1)
    mu, mv = core.compute(3, 4)
    wu, wv = oracle.peel(nU, nV, off, adj, 3, 4)
    assert np.array_equal(mu.cpu().numpy(), wu) and np.array_equal(mv.cpu().numpy(), wv)
    assert (core.stats()["launches"] > 1) == ((name, value) in KERNELS + PEEL)
    _check(core, nU, nV, off, adj, [(1, 2), (2, 2), (2, 5), (4, 3)], (name, value) in KERNELS + CHAINS)
    core.close()


@pytest.mark.parametrize("nalpha", [1, 4, 5, 8, 9, 13, 16, 17, 40])
@pytest.mark.parametrize("packed", [1, 0])
def test_chains_of_every_width(small, nalpha, packed):
    nU, nV, eu, ev, off, adj = small
    core = ABCore(0)
    core.load_edges(nU, nV, eu.cuda(), ev.cuda())
    core.set_param("small_peel", 0)
    core.set_param("packed_counts", packed)
    pairs = [(a, b) for a in range(nalpha) for b in (0, 1, 2, 4, 9)]
    np.random.default_rng(nalpha).shuffle(pairs)
    _check(core, nU, nV, off, adj, [tuple(int(x) for x in p) for p in pairs], True)
    core.close()


def test_a_degree_that_needs_32_bit_counts():
    nU, nV = 70_003, 301
    eu, ev = synth.chung_lu_edges(nU, 300, 300_000, 2.3, 2.2, 7)
    eu, ev = eu.numpy(), ev.numpy()
    eu = np.concatenate([eu, np.arange(nU, dtype=np.int32)])  # one vertex of the lower layer has every upper one
    ev = np.concatenate([ev, np.full(nU, 300, dtype=np.int32)])
    off, adj = oracle.build_csr(nU, nV, eu, ev)
    core = ABCore(0)
    core.load_edges(nU, nV, torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda())
    _check(core, nU, nV, off, adj, [(a, b) for a in (1, 2, 3, 6, 20) for b in (1, 50, 3000, 65535, 65536, 70003)], True)
    core.close()


def test_a_captured_plan_serves_any_buffers(small):
    nU, nV, eu, ev, off, adj = small
    core = ABCore(0)
    core.load_edges(nU, nV, eu.cuda(), ev.cuda())
    core.set_param("small_peel", 0)
    pairs = synth.grid_pairs(6, 1, 40)
    a, b = [p[0] for p in pairs], [p[1] for p in pairs]
    want = [oracle.peel(nU, nV, off, adj, *p) for p in pairs]
    for shift in (0, 0, 1, 4):  # (odd addresses take the byte stores)
        mu = torch.full((len(pairs) * nU + shift,), 7, dtype=torch.uint8, device="cuda")[shift:].view(len(pairs), nU)
        mv = torch.full((len(pairs) * nV + shift,), 7, dtype=torch.uint8, device="cuda")[shift:].view(len(pairs), nV)
        core.compute_batch(a, b, mu, mv)
        for k, (wu, wv) in enumerate(want):
            assert np.array_equal(mu[k].cpu().numpy(), wu) and np.array_equal(mv[k].cpu().numpy(), wv), (shift, pairs[k])
    core.close()


def test_more_pairs_than_one_launch_writes(small):
    # many pairs given again and again: a wave's masks take several launches
    nU, nV, eu, ev, off, adj = small
    core = ABCore(0)
    core.load_edges(nU, nV, eu.cuda(), ev.cuda())
    core.set_param("small_peel", 0)
    distinct = [(a, b) for a in range(1, 17) for b in (1, 2, 3, 5, 8, 13)]
    rng = np.random.default_rng(3)
    at = np.concatenate([rng.integers(0, len(distinct), 30_000), np.arange(len(distinct))])
    want = [oracle.peel(nU, nV, off, adj, *p) for p in distinct]
    wu, wv = (torch.from_numpy(np.stack([w[k] for w in want])).cuda() for k in (0, 1))
    for shift in (0, 1):
        mu = torch.full((len(at) * nU + shift,), 7, dtype=torch.uint8, device="cuda")[shift:].view(len(at), nU)
        mv = torch.full((len(at) * nV + shift,), 7, dtype=torch.uint8, device="cuda")[shift:].view(len(at), nV)
        core.compute_batch([distinct[k][0] for k in at], [distinct[k][1] for k in at], mu, mv)
        idx = torch.from_numpy(at).cuda()
        assert torch.equal(mu, wu[idx]) and torch.equal(mv, wv[idx])
    core.close()
