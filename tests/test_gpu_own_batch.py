"""The batch tests on the transition-table kernel, and batches whose instances
use both kernels, large ones of either split into parts."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from tests.pinned_plans import PINNED, own_scans  # noqa: E402, F401
from tests.test_gpu_batch import (  # noqa: E402, F401
    BASE_N, _check, _oracle_results, base, d_base, mixed, pm, pytestmark, synth, test_batch_capacity_short,
    test_batch_equals_plain_single_scans, test_batch_every_warp_count_and_graph_replay,
    test_batch_large_tables_hybrid, test_batch_matches_oracle_per_instance, test_batch_splits_large_instances,
    test_pm_scan_batch_host_call_against_oracle)


@pytest.mark.parametrize("warps,placement", [(8, 0), (12, 1), (16, 0)])
def test_both_kernels_in_one_batch(base, d_base, warps, placement):
    """Every other instance keeps its automaton; two of each kind are split."""
    Ps, off, ln = [], [], []
    for j in range(24):
        o = j * 300_000 + 7 * j
        n = 2_500_000 + 13 * j if j < 4 else 900 * j + j
        Ps.append(synth.batch_patterns(base[:BASE_N], o, n, 40 * (j + 1), 8 + j, 1200 + j))
        off.append(o), ln.append(min(n, BASE_N - o))
    grams = [pm.PatternSet(pm.pm_ac_compile(P, None), pm.PM_ALGO_AC) if j % 2 else pm.PatternSet.ac(P, dict(PINNED))
             for j, P in enumerate(Ps)]
    assert [s.scan_kind() != pm.PM_SCAN_METHOD for s in grams] == [bool(j % 2) for j in range(24)]
    off, ln = np.array(off, np.int64), np.array(ln, np.int64)
    want = _oracle_results(base, Ps, off, ln)
    b = pm.Batch.exact(grams, d_base, off, ln)
    b.set_warps(warps)
    b.set_placement(placement)
    b.scan()
    assert b.status() == pm.PM_OK
    _check(b.results(), want, "both kernels")
    b.capture()
    for rep in range(2):
        b.occ.fill_(-1)
        b.counts.fill_(-1)
        b.replay()
        assert b.status() == pm.PM_OK
        _check(b.results(), want, f"both kernels, replay {rep}")
    c = pm.Batch(grams, d_base, off, ln, None)
    c.set_warps(warps)
    c.scan()
    assert c.status() == pm.PM_OK
    for j, ((_, cnt, tot), (wo, wc)) in enumerate(zip(c.results(), want)):
        assert tot == wo.size and np.array_equal(cnt, wc), f"counts-only instance {j}"
    for x in (b, c, *grams):
        x.close()
