"""Parameters that follow a rule until they are set: the rule can be asked for again, and reading every parameter and
writing it back changes nothing that a query does."""

import pytest

import synth
from paper_2606_07148_gb300 import ABCore, ABCoreError

pytestmark = pytest.mark.gpu

RULED = ("round0", "round0_variant", "flush_steps")
NAMES = ("chunk", "grab_div", "local_rounds", "batch_entries_small", "batch_entries", "flush_steps", "packed_counts", "round0",
         "round0_variant", "round0_hub", "count_swizzle", "pdl", "blocks_per_sm", "mode", "timeout_ms", "emit_scatter_max_pct",
         "emit_bitmap_min_pct", "probe_bytes", "batch_wave", "hub_degree", "timing", "timing_kinds", "serve_inserts", "algo",
         "query_scope", "batch_seed", "batch_plain_below", "log_level", "small_peel")


def _what(core, pairs):
    core.set_param("reset_stats", 1)
    for a, b in pairs:
        core.compute(a, b)
    core.compute_batch([p[0] for p in pairs], [p[1] for p in pairs])
    st = core.stats()
    return st["launches"], st["round0_rows"], st["mode"], st["grid_blocks"]


def test_reading_and_writing_back_changes_nothing():
    # a small graph (one-block kernels) and one whose first rounds are long enough to be walked by rule
    for nU, nV, m, pairs in ((2000, 1500, 20000, [(2, 3), (5, 5)]), (1_500_001, 750_003, 30_000_000, [(40, 40), (300, 300)])):
        eu, ev = synth.chung_lu_edges(nU, nV, m, 2.1, 2.3, 5, device="cuda")
        core = ABCore(0)
        core.load_edges(nU, nV, eu, ev)
        before = _what(core, pairs)
        read = {k: core.get_param(k) for k in NAMES}
        for k, v in read.items():
            core.set_param(k, v)
        assert _what(core, pairs) == before
        assert {k: core.get_param(k) for k in NAMES} == read
        assert all(read[k] == -1 for k in RULED)
        assert m < 1_000_000 or before[1] > 0  # (the rule walks)
        core.close()


def test_a_rule_can_be_asked_for_again():
    core = ABCore(0)
    eu, ev = synth.chung_lu_edges(1_500_001, 750_003, 30_000_000, 2.1, 2.3, 5, device="cuda")
    core.load_edges(1_500_001, 750_003, eu, ev)
    wave = core.get_param("batch_wave")
    before = _what(core, [(40, 40)])
    for k, v in (("round0", 0), ("round0_variant", 2), ("flush_steps", 1), ("batch_wave", 2)):
        core.set_param(k, v)
        assert core.get_param(k) == v
    assert _what(core, [(40, 40)])[1] == 0
    for k in RULED + ("batch_wave",):
        core.set_param(k, -1)
        assert core.get_param(k) == (wave if k == "batch_wave" else -1)
        with pytest.raises(ABCoreError):
            core.set_param(k, -2)
    assert _what(core, [(40, 40)]) == before
    core.close()
