"""The gram scans on long runs of one byte: of a letter, and of a byte outside
the alphabet that has a letter's code (N that of G), beside sets with grams of
that letter only."""
import os

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # collected on CPU-only machines, never run there
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1407_2889_gb300 import pmscan as pm  # noqa: E402

THREADS = os.cpu_count() or 4
RUNS = b"NNNGTAnN\n\0"


def _text(rng, A, n):
    T = A[rng.integers(0, A.size, n)]
    at = 0
    while at < n:
        at += int(rng.integers(1, 3000))
        ln = int(rng.integers(1, 5000)) if rng.random() < 0.7 else int(rng.integers(1, 40))
        T[at:at + ln] = RUNS[int(rng.integers(0, len(RUNS)))]
        at += ln
    return T


@pytest.mark.parametrize("alphabet", [b"ACGT", b"acgt", b"GT"])
@pytest.mark.parametrize("m", [5, 8, 10, 12, 17, 32])
def test_runs(alphabet, m):
    A = np.frombuffer(alphabet, np.uint8)
    rng = np.random.default_rng(m + len(alphabet))
    T = _text(rng, A, 150_001)
    d = min(60, 2 ** m)
    P = A[rng.integers(0, A.size, (d, m))]
    for k, c in enumerate(alphabet):
        P[k] = c
        P[k + 5, :m - 1] = c
        P[k + 10, 1:] = c
    V = [bytes(r[:max(4, m - k % 4)]) for k, r in enumerate(P)]
    want, want_var = oracle.dictionary(T, P, threads=THREADS), oracle.dictionary_var(T, V, threads=THREADS)
    buf = torch.from_numpy(np.concatenate([np.zeros(16, np.uint8), T])).cuda()
    for off in (16, 13):
        d_text = buf[off:off + T.size]
        d_text.copy_(torch.from_numpy(T))
        for make, P_, w in ((pm.PatternSet.ac, P, want), (pm.PatternSet.pfac, P, want),
                            (lambda x: pm.PatternSet.wm(x, 2), P, want), (pm.PatternSet.acv, V, want_var),
                            (lambda x: pm.PatternSet.wmv(x, 2), V, want_var)):
            s = make(P_)
            occ, cnt = s.scan(d_text)
            assert np.array_equal(occ, w[0]) and np.array_equal(cnt, w[1])
            assert np.array_equal(s.scan(d_text, counts_only=True)[1], w[1])
            s.close()
    s = pm.PatternSet.ac(P)   # the batched form
    offs, lens = [0, 16, 1600, 40000], [T.size, 60000, 2561, 100001]
    b = pm.Batch.exact([s] * 4, torch.from_numpy(T).cuda(), offs, lens)
    b.scan()
    assert b.status() == pm.PM_OK
    for (occ, cnt, tot), o, n in zip(b.results(), offs, lens):
        w = oracle.dictionary(T[o:o + n], P, threads=THREADS)
        assert tot == w[0].size and np.array_equal(occ, w[0]) and np.array_equal(cnt, w[1])
    b.close()
    s.close()
