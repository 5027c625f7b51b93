"""Working memory a context keeps between calls: batches into other buffers than the plan was
captured with, graphs of changing sizes loaded in turn, and every kind of call after each."""

import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2606_07148_gb300 import ABCore

pytestmark = pytest.mark.gpu


def _masks(nU, nV, off, adj, pairs):
    w = [oracle.peel(nU, nV, off, adj, a, b) for a, b in pairs]
    return np.stack([x[0] for x in w]), np.stack([x[1] for x in w])


def test_batch_plan_serves_any_output_buffers():
    nU, nV, eu, ev = synth.make_graph("peel-2000x1500-20k")
    off, adj = oracle.build_csr(nU, nV, eu.numpy(), ev.numpy())
    pairs = [(a, b) for a in (1, 3, 6) for b in (2, 4, 9)]
    wu, wv = _masks(nU, nV, off, adj, pairs)
    core = ABCore(0)
    core.load_edges(nU, nV, eu.cuda(), ev.cuda())
    outs = []
    for k in range(4):  # the last pair of buffers is misaligned for 4-byte stores
        du = torch.full((len(pairs) * nU + k,), 7, dtype=torch.uint8, device="cuda")[k:].view(len(pairs), nU)
        dv = torch.full((len(pairs) * nV + k,), 7, dtype=torch.uint8, device="cuda")[k:].view(len(pairs), nV)
        core.compute_batch([p[0] for p in pairs], [p[1] for p in pairs], du, dv)
        outs.append((du, dv))
    for du, dv in outs:
        assert np.array_equal(du.cpu().numpy(), wu) and np.array_equal(dv.cpu().numpy(), wv)
    core.close()


def test_graphs_of_changing_sizes_in_one_context():
    rng = np.random.default_rng(2)
    core = ABCore(0)
    for nU, nV, m in [(3000, 2000, 30000), (50, 40, 200), (40000, 9000, 200000), (3001, 1999, 30001), (50, 40, 0)]:
        key = rng.choice(nU * nV, m, replace=False)
        eu, ev = (key // nV).astype(np.int32), (key % nV).astype(np.int32)
        off, adj = oracle.build_csr(nU, nV, eu, ev)
        core.load_edges(nU, nV, torch.from_numpy(eu).cuda(), torch.from_numpy(ev).cuda())
        wu, wv = _masks(nU, nV, off, adj, [(3, 4), (4, 9)])
        mu, mv = core.compute(3, 4)
        bu, bv = core.compute_batch([3, 4], [4, 9])
        lab, nc = oracle.components(nU, nV, off, adj)
        lu, lv, got = core.components()
        cu, cv, _ = core.core_numbers()
        want = oracle.core_numbers(nU, nV, off, adj)
        assert np.array_equal(mu.cpu().numpy(), wu[0]) and np.array_equal(mv.cpu().numpy(), wv[0])
        assert np.array_equal(bu.cpu().numpy(), wu) and np.array_equal(bv.cpu().numpy(), wv)
        assert got == nc and np.array_equal(np.concatenate([lu.cpu().numpy(), lv.cpu().numpy()]), lab)
        assert np.array_equal(np.concatenate([cu.cpu().numpy(), cv.cpu().numpy()]), want)
    assert core.stats()["device_bytes"] < 1 << 30
    core.close()
