"""GPU parity of the sampled-gram scan where it can go wrong: texts that end
inside a row, a batch or a tile, unaligned texts, bytes outside the alphabet,
every stride, list and counts, and texts in which every gram passes."""
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


def _check(s, T, want, off=0):
    buf = torch.zeros(T.size + 16, dtype=torch.uint8, device="cuda")
    d_text = buf[off:off + T.size]
    d_text.copy_(torch.from_numpy(T))
    occ, cnt = s.scan(d_text)
    assert np.array_equal(occ, want[0]) and np.array_equal(cnt, want[1])
    assert np.array_equal(s.scan(d_text, counts_only=True)[1], want[1])


@pytest.mark.parametrize("alphabet", [b"ACGT", b"ACDEFGHIKLMNPQRSTVWY"])
@pytest.mark.parametrize("m", [4, 8, 9, 10, 13, 16, 20, 31, 65])
def test_text_ends(alphabet, m):
    rng = np.random.default_rng(41 + m)
    A = np.frombuffer(alphabet, np.uint8)
    base = A[rng.integers(0, A.size, 40000)]
    base[rng.integers(0, base.size, 300)] = ord("N")
    P = A[rng.integers(0, A.size, (90, m))]
    for r in range(0, 90, 2):
        P[r] = base[r * 37:r * 37 + m]
    P[5] = P[4]
    s = pm.PatternSet.ac(P)
    for n in (m, 511, 512, 513, 2047, 3072, 3073, 4096 + 15, 8192, 24575, 40000):
        T = base[:n].copy()
        T[n - m:] = P[4]  # an occurrence at the very end
        for off in (0, 1, 6):
            _check(s, T, oracle.dictionary(T, P, threads=THREADS), off)
    s.close()


@pytest.mark.parametrize("m", [8, 16, 32])
def test_every_gram_passes(m):
    T = np.full(70001, ord("A"), np.uint8)
    P = np.full((3, m), ord("A"), np.uint8)
    P[2, -1] = ord("C")
    want = oracle.dictionary(T, P, threads=THREADS)
    for s in (pm.PatternSet.ac(P), pm.PatternSet.wm(P, 2), pm.PatternSet.pfac(P)):
        _check(s, T, want)
        s.close()
    V = [b"A" * k for k in range(max(4, m - 12), m + 1)]
    want = oracle.dictionary_var(T, V, threads=THREADS)
    for s in (pm.PatternSet.acv(V), pm.PatternSet.wmv(V, 2)):
        _check(s, T, want)
        s.close()


@pytest.mark.parametrize("d,m", [(40000, 12), (70000, 24), (20000, 40)])
def test_wide_codes_and_device_counters(d, m):
    rng = np.random.default_rng(d)
    A = np.frombuffer(b"ACGT", np.uint8)
    T = A[rng.integers(0, 4, 300000)]
    P = A[rng.integers(0, 4, (d, m))]
    P[::3] = T[(np.arange(0, d, 3) * 4)[:, None] + np.arange(m)[None, :]]
    P[1] = P[0]
    s = pm.PatternSet.ac(P)
    want = oracle.dictionary(T, P, threads=THREADS)
    _check(s, T, want)
    # the batched form, whole and split, next to a small text
    d_text = torch.from_numpy(T).cuda()
    b = pm.Batch.exact([s, s], d_text, [0, 16], [T.size, 5000])
    b.scan()
    got = b.results()
    small = oracle.dictionary(T[16:5016], P, threads=THREADS)
    for g, w in zip(got, (want, small)):
        assert np.array_equal(g[0], w[0]) and np.array_equal(g[1], w[1])
    b.close()
    s.close()


@pytest.mark.parametrize("m", [8, 20])
def test_captured_in_a_graph(m):
    """A scan's dependent launches captured and replayed over changing texts."""
    rng = np.random.default_rng(m)
    A = np.frombuffer(b"ACGT", np.uint8)
    P = A[rng.integers(0, 4, (200, m))]
    n = 50000
    s = pm.PatternSet.ac(P)
    d_text = torch.zeros(n, dtype=torch.uint8, device="cuda")
    counts = torch.zeros(200, dtype=torch.int64, device="cuda")
    occ = torch.zeros(n, dtype=torch.int64, device="cuda")
    n_occ = torch.zeros(1, dtype=torch.int64, device="cuda")
    ws = torch.empty(s.workspace_bytes(n), dtype=torch.uint8, device="cuda")
    side = torch.cuda.Stream()

    def scan():
        pm.pm_scan_device(s.h, d_text, n, 0, counts, occ, n, n_occ, ws, ws.numel(), torch.cuda.current_stream())

    with torch.cuda.stream(side):
        scan()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        scan()
    for k in range(3):
        T = A[rng.integers(0, 4, n)]
        T[k * 700:k * 700 + m] = P[k]
        d_text.copy_(torch.from_numpy(T))
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        want = oracle.dictionary(T, P, threads=THREADS)
        tot = int(n_occ.item())
        assert tot == want[0].size
        assert np.array_equal(occ[:tot].cpu().numpy().view(np.uint64), want[0])
        assert np.array_equal(counts.cpu().numpy(), want[1])
    s.close()
