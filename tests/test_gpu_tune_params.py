"""What pm_tune returns: the same patterns compiled with it take the scan that
the tuned set takes, also where the method's own scan beats the grams (a text
of one letter against patterns that begin with a run of it)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU-only machines, never run there
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1407_2889_gb300 import pmscan as pm  # noqa: E402


@pytest.mark.parametrize("run", [True, False])
@pytest.mark.parametrize("d,m", [(40, 32), (60, 24), (100, 40), (200, 8)])
@pytest.mark.parametrize("make", [pm.PatternSet.ac, lambda P, p=None: pm.PatternSet.wm(P, 4, p)])
def test_returned_parameters_name_the_winner(make, d, m, run):
    A = np.frombuffer(b"ACGT", np.uint8)
    rng = np.random.default_rng(d + m)
    P = A[rng.integers(0, 4, (d, m))]
    P[:, :2 * m // 3] = ord("A")
    T = np.full(4 << 20, ord("A"), np.uint8) if run else A[rng.integers(0, 4, 4 << 20)]
    d_text = torch.from_numpy(T).cuda()
    for counts_only in (False, True):
        s = make(P)
        first = s.scan_kind()
        for _ in range(2):   # the second time from the tuned parameters
            best, _ms = s.tune(d_text, counts_only=counts_only, reps=2)
            r = make(P, best)
            assert r.scan_kind() == s.scan_kind(), best
            automatic = best["stride"] < 2 and not any(
                best[k] for k in ("placement", "warps_per_cta", "ctas_per_sm", "counters", "ids_place"))
            assert not automatic or s.scan_kind() == first, best
            a, b = s.scan(d_text), r.scan(d_text)
            assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
            r.close()
        s.close()
