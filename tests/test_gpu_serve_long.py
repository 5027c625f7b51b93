"""A served update whose re-peel takes longer than every wait of the loop is waited for: the waits end when nothing
gets on any more, not when one update is long."""

import time

import numpy as np
import pytest

from paper_2606_07148_gb300 import ABCore, abi

pytestmark = pytest.mark.gpu


def test_a_cascade_and_a_region_longer_than_the_limit():
    # a cycle is its own (2,2)-core; without one edge all of it falls, two vertices a level, and comes back the same way
    k = 400_000
    i = np.arange(k, dtype=np.int32)
    eu, ev = np.concatenate([i, (i + 1) % k]), np.concatenate([i, i])
    core = ABCore(0)
    core.load_edges(k, k, eu, ev)
    core.set_param("timeout_ms", 1)  # (the loop's own waits: 1 ms past its idle spell of 200)
    core.serve_start([(2, 2)], ring_slots=8)
    ops = [abi.ABCORE_DELETE, abi.ABCORE_INSERT, abi.ABCORE_DELETE]
    reqs = (abi.abcore_req * 3)(*[abi.abcore_req(op, 7, 7, 0, 10 + j) for j, op in enumerate(ops)])
    assert core.serve_submit(reqs) is not None
    out, t0, first = [], time.time(), None
    while len(out) < 3:
        out.extend(core.serve_poll(16))
        if out and first is None:
            first = time.time() - t0
        assert time.time() - t0 < 60
    core.set_param("timeout_ms", 4000)
    core.serve_stop()
    assert first > 0.25, "the cascade is too short for this test: %.3f s" % first
    assert [(r.tag, r.status, r.in_core) for r in out] == [(10, 0, 0), (11, 0, 1), (12, 0, 0)]
    mu, mv = core.compute(2, 2)
    assert int(mu.sum()) == 0 and int(mv.sum()) == 0
    core.close()
