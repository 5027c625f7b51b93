"""Little device memory left: the blocks a context keeps go back when one of its allocations would fail without them, and a
query whose walked first round has no room for its list queues it instead."""

import gc

import numpy as np
import pytest
import torch

import oracle
import synth
from paper_2606_07148_gb300 import ABCore, ABCoreError, abi

pytestmark = pytest.mark.gpu


def _fill(keep):
    """Take all free device memory but about `keep` bytes."""
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = []
    while True:
        n = torch.cuda.mem_get_info()[0] - keep
        if n < 4 << 20:
            return held
        try:
            held.append(torch.empty(n if not held else min(n, 64 << 20), dtype=torch.uint8, device="cuda"))
        except torch.cuda.OutOfMemoryError:
            if held:
                return held
            keep += 64 << 20


def _equal(core, nU, nV, off, adj, pair):
    wu, wv, _ = oracle.peel_many(nU, nV, off, adj, [pair])[pair]
    mu, mv = core.compute(*pair, np.empty(nU, np.uint8), np.empty(nV, np.uint8))
    return np.array_equal(mu, wu) and np.array_equal(mv, wv)


def test_kept_blocks_go_back():
    one, two = (1_500_001, 750_003, 30_000_000), (1_200_001, 600_003, 24_000_000)
    eu, ev = synth.chung_lu_edges(*one, 2.1, 2.3, seed=5, device="cuda")
    fu, fv = (x.clone() for x in synth.chung_lu_edges(*two, 2.1, 2.3, seed=6, device="cuda"))
    off, adj = oracle.build_csr(two[0], two[1], fu.cpu().numpy(), fv.cpu().numpy())
    core = ABCore(0)
    wu, wv = synth.chung_lu_edges(300_000, 150_000, 6_000_000, 2.1, 2.3, seed=7, device="cuda")
    core.load_edges(300_000, 150_000, wu, wv)  # (every kernel's code is on the device before memory is short)
    core.compute(40, 40, np.empty(300_000, np.uint8), np.empty(150_000, np.uint8))
    core.load_edges(one[0], one[1], eu, ev)
    before = core.stats()["device_bytes"]
    held = _fill(48 << 20)
    try:
        # the second graph's arrays fit none of the first's blocks: its load has to give them back
        core.load_edges(two[0], two[1], fu, fv)
        assert _equal(core, two[0], two[1], off, adj, (40, 40))
        assert core.stats()["device_bytes"] < before
    finally:
        del held
        core.close()
        torch.cuda.empty_cache()


def test_a_walk_without_room_for_its_list_is_queued():
    nU, nV, eu, ev = synth.make_graph("peel-4Mx2M-80M", device="cuda")
    off, adj = oracle.build_csr(nU, nV, eu.cpu().numpy(), ev.cpu().numpy())
    core = ABCore(0)
    core.load_edges(nU, nV, eu, ev)
    del eu, ev
    pair = (3, 50)  # 3.8M candidates, 60 MB of list
    core.compute(50, 50, np.empty(nU, np.uint8), np.empty(nV, np.uint8))  # (walked: the kernels are loaded, the list is 6 MB)
    core.set_param("round0", 0)
    assert _equal(core, nU, nV, off, adj, pair)
    core.set_param("round0", -1)
    held = _fill(24 << 20)
    try:
        with pytest.raises(ABCoreError) as e:  # (fails, and gives the kept blocks back)
            core.measure_atomics(4 << 30)
        assert e.value.code == abi.ABCORE_ENOMEM
        held += _fill(24 << 20)
        core.set_param("reset_stats", 1)
        assert _equal(core, nU, nV, off, adj, pair)
        assert core.stats()["round0_rows"] == 0
        core.set_param("round0", 1)  # (asked for, it is not passed over)
        with pytest.raises(ABCoreError) as e:
            core.compute(*pair, np.empty(nU, np.uint8), np.empty(nV, np.uint8))
        assert e.value.code == abi.ABCORE_ENOMEM
        core.set_param("round0", -1)
        assert _equal(core, nU, nV, off, adj, (50, 50))
    finally:
        del held
        torch.cuda.empty_cache()
    core.set_param("reset_stats", 1)
    assert _equal(core, nU, nV, off, adj, pair)
    assert core.stats()["round0_rows"] > 0
    core.close()
