"""The serving loop's hand-over between its warps: answers equal the oracle's replay whatever the ring,
the batch and the number of targets, for edges that come and go many times (their segments grow and
fill with deleted entries), rows the edge search cuts once, several times or not at all, and both block sizes."""

import time

import numpy as np
import pytest

import oracle
from paper_2606_07148_gb300 import ABCore, abi

pytestmark = pytest.mark.gpu


def _graph(rng):
    # two hub rows (searched in several cuts), ordinary rows, and vertices without edges
    key = {(0, j) for j in range(1500)} | {(i, 3) for i in range(1, 1200)}
    key |= {(int(u), int(v)) for u, v in zip(rng.integers(2, 400, 4000), rng.integers(0, 300, 4000))}
    e = np.array(sorted(key), dtype=np.int32)
    return 1210, 1510, np.ascontiguousarray(e[:, 0]), np.ascontiguousarray(e[:, 1])


def _ops(rng, n, nU, nV, eu, ev):
    """Updates over a small pool of pairs, present or not: many repeats, so EEXIST and ENOENT too."""
    pool = [(int(eu[k]), int(ev[k])) for k in rng.integers(0, len(eu), 60)]
    pool += [(int(u), int(v)) for u, v in zip(rng.integers(0, 40, 60), rng.integers(0, 40, 60))]
    pool += [(0, int(v)) for v in rng.integers(1490, nV, 20)] + [(int(u), 3) for u in rng.integers(1190, nU, 20)]
    at = rng.integers(0, len(pool), n)
    return rng.integers(0, 2, n).astype(np.int8), np.array([pool[k][0] for k in at], np.int32), np.array([pool[k][1] for k in at], np.int32)


@pytest.mark.parametrize("ntargets,ring,batch,n", [(1, 5, 3, 400), (3, 64, 64, 1500), (3, 1024, 500, 3000), (2, 1024, 1, 200),
                                                   (160, 256, 100, 300)])
def test_answers_equal_the_replay(ntargets, ring, batch, n):
    rng = np.random.default_rng(ntargets + ring)
    nU, nV, eu, ev = _graph(rng)
    targets = [(1 + t % 13, 1 + (t // 13) % 14) for t in range(ntargets)] if ntargets > 3 else [(6, 8), (2, 2), (9, 12)][:ntargets]
    op, u, v = _ops(rng, n, nU, nV, eu, ev)
    tg = rng.integers(0, ntargets, n)
    al, be = np.array([targets[t][0] for t in tg], np.int32), np.array([targets[t][1] for t in tg], np.int32)
    ans, bits, status = oracle.replay(nU, nV, eu, ev, op, u, v, al, be)
    core = ABCore(0)
    core.set_param("serve_inserts", 16)  # pools fill and grow on the way
    core.load_edges(nU, nV, eu, ev)
    core.serve_start(targets, ring_slots=ring)
    out, k, t0 = [], 0, time.time()
    while len(out) < n:
        assert time.time() - t0 < 60, "stalled: %d submitted, %d answered" % (k, len(out))
        if k < n:
            hi = min(n, k + batch)
            reqs = (abi.abcore_req * (hi - k))(*[abi.abcore_req(int(op[i]), int(u[i]), int(v[i]), int(tg[i]), i) for i in range(k, hi)])
            if core.serve_submit(reqs) is not None:
                k = hi
        out.extend(core.serve_poll(4096))
        if batch == 1 and k < n and rng.random() < 0.02:
            time.sleep(0.25)  # past the idle spell: the loop leaves and is launched again
    core.serve_stop()
    assert [r.tag for r in out] == list(range(n))
    assert np.array_equal(np.array([r.status for r in out]), status)
    assert np.array_equal(np.array([r.in_core for r in out]), ans)
    assert np.array_equal(np.array([r.u_in | (r.v_in << 1) for r in out]), bits)
    # the updates are in the graph: components as the oracle finds them
    cur = set(zip(eu.tolist(), ev.tolist()))
    for i in range(n):
        if status[i] == 0:
            (cur.add if op[i] == 0 else cur.discard)((int(u[i]), int(v[i])))
    e = np.array(sorted(cur), dtype=np.int32)
    off, adj = oracle.build_csr(nU, nV, np.ascontiguousarray(e[:, 0]), np.ascontiguousarray(e[:, 1]))
    want, wn = oracle.components(nU, nV, off, adj)
    lu, lv, nc = core.components()
    assert nc == wn and np.array_equal(np.concatenate([lu.cpu().numpy(), lv.cpu().numpy()]), want)
    core.close()
