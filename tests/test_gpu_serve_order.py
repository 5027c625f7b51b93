"""Requests reach every lane of the serving loop as the host published them: bursts of every length from one to more
than a warp, published while the loop polls, through rings whose slots are reused all the time."""

import time

import numpy as np
import pytest

import oracle
from paper_2606_07148_gb300 import ABCore, abi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ring,ntargets", [(37, 1), (64, 4), (200, 2)])
def test_bursts_through_reused_slots(ring, ntargets):
    rng = np.random.default_rng(ring)
    nU, nV = 300, 200
    key = {(int(a), int(b)) for a, b in zip(rng.integers(0, nU, 2500), rng.integers(0, nV, 2500))}
    e = np.array(sorted(key), dtype=np.int32)
    eu, ev = np.ascontiguousarray(e[:, 0]), np.ascontiguousarray(e[:, 1])
    targets = [(4, 5), (2, 2), (7, 9), (1, 12)][:ntargets]
    bursts = [b for b in range(1, 36) for _ in range(3)]
    rng.shuffle(bursts)
    n = sum(bursts)
    op = rng.integers(0, 2, n).astype(np.int8)
    u, v = rng.integers(0, nU, n).astype(np.int32), rng.integers(0, nV, n).astype(np.int32)
    tg = rng.integers(0, ntargets, n)
    al, be = np.array([targets[t][0] for t in tg], np.int32), np.array([targets[t][1] for t in tg], np.int32)
    ans, bits, status = oracle.replay(nU, nV, eu, ev, op, u, v, al, be)
    core = ABCore(0)
    core.load_edges(nU, nV, eu, ev)
    core.serve_start(targets, ring_slots=ring)
    out, k, t0 = [], 0, time.time()
    for b in bursts:
        reqs = (abi.abcore_req * b)(*[abi.abcore_req(int(op[i]), int(u[i]), int(v[i]), int(tg[i]), 7 * i) for i in range(k, k + b)])
        while core.serve_submit(reqs) is None:
            out.extend(core.serve_poll(5))
            assert time.time() - t0 < 60
        k += b
    while len(out) < n:
        out.extend(core.serve_poll(4096))
        assert time.time() - t0 < 60
    core.serve_stop()
    assert [r.tag for r in out] == [7 * i for i in range(n)]
    assert np.array_equal(np.array([r.status for r in out]), status)
    assert np.array_equal(np.array([r.in_core for r in out]), ans)
    assert np.array_equal(np.array([r.u_in | (r.v_in << 1) for r in out]), bits)
    core.close()
