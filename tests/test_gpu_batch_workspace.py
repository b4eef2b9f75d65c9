"""A batch plan that needs a larger workspace than the prepared one: scans
refuse the smaller buffer, and run in one of the new size."""
import os

import numpy as np
import pytest

import oracle
from paper_1407_2889_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU-only machines, never run there
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1407_2889_gb300 import pmscan as pm  # noqa: E402


def test_one_warp_needs_more_parts():
    T = synth.est_text(200_000, 3)
    P = synth.batch_patterns(T, 0, T.size, 60, 12, 5)
    d_text = torch.from_numpy(T).cuda()
    s = pm.PatternSet.ac(P, {"ids_place": 1})   # a pinned plan: the transition-table kernel, split by warps
    b = pm.Batch.exact([s], d_text, [0], [T.size])
    before = pm.pm_batch_workspace_bytes(b.b)
    small = b._bufs()
    pm.pm_batch_set_warps(b.b, 1)
    assert pm.pm_batch_workspace_bytes(b.b) > before
    for call in (lambda: pm.pm_batch_scan_device(b.b, *small), lambda: pm.pm_batch_tune(b.b, *small, reps=1),
                 lambda: pm.pm_batch_capture(b.b, *small)):
        with pytest.raises(pm.PmError) as e:
            call()
        assert e.value.code == pm.PM_EINVAL
    b.set_warps(1)
    b.scan()
    assert b.status() == pm.PM_OK
    occ, cnt, tot = b.results()[0]
    want = oracle.dictionary(T, P, threads=os.cpu_count() or 4)
    assert tot == want[0].size and np.array_equal(occ, want[0]) and np.array_equal(cnt, want[1])
    b.close()
    s.close()
