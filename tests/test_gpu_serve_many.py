"""Several serving targets an SM run at the same time: none waits for another's idle spell."""

import time

import numpy as np
import pytest

from paper_2606_07148_gb300 import ABCore, abi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per_sm", [1, 2, 4, 5])
def test_every_target_answers_before_an_idle_spell_has_passed(per_sm):
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    nt = per_sm * sms - 3
    rng = np.random.default_rng(per_sm)
    key = np.unique(rng.integers(0, 60 * 50, 1200))
    eu, ev = (key // 50).astype(np.int32), (key % 50).astype(np.int32)
    core = ABCore(0)
    core.set_param("serve_inserts", 64)
    core.load_edges(60, 50, eu, ev)
    core.serve_start([(1 + t % 20, 1 + t // 20) for t in range(nt)], ring_slots=nt)
    # one update for every target, the same edge out and in again
    reqs = (abi.abcore_req * nt)(*[abi.abcore_req(abi.ABCORE_DELETE if t % 2 == 0 else abi.ABCORE_INSERT, int(eu[0]), int(ev[0]), t, t)
                                   for t in range(nt)])
    took = []
    for _ in range(2):  # (the first launch of the kernel loads its code)
        t0, out = time.time(), []
        assert core.serve_submit(reqs) is not None
        while len(out) < nt:
            out.extend(core.serve_poll(4096))
            assert time.time() - t0 < 60
        took.append(time.time() - t0)
        # an odd count leaves the edge out: put it back
        if nt % 2:
            back = (abi.abcore_req * 1)(abi.abcore_req(abi.ABCORE_INSERT, int(eu[0]), int(ev[0]), 0, nt))
            assert core.serve_submit(back) is not None
            while not core.serve_poll(1):
                assert time.time() - t0 < 60
        assert all(r.status == 0 for r in out)
        time.sleep(0.3)  # (the loop leaves)
    core.serve_stop()
    core.close()
    assert took[1] < 0.19, took
