"""The sampled-gram tables without a GPU: a host walk of them gives the
oracle's occurrences, already in (i, r) order, for every stride and gram form
the planner picks, and pinned launch plans get no such tables."""
import os

import numpy as np
import pytest

import oracle
from paper_1407_2889_gb300 import pmscan as pm

HOST = {"host_only": 1}
THREADS = os.cpu_count() or 4


def _text(rng, alphabet, n, noise=b"N\n"):
    A = np.frombuffer(alphabet, np.uint8)
    T = A[rng.integers(0, A.size, n)]
    if n > 8:
        T[rng.integers(0, n, n // 50)] = np.frombuffer(noise, np.uint8)[rng.integers(0, len(noise), n // 50)]
        T[n // 2: n // 2 + min(200, n // 4)] = A[0]  # a run of one letter
    return T


def _rows(rng, T, alphabet, d, m):
    A = np.frombuffer(alphabet, np.uint8)
    P = A[rng.integers(0, A.size, (d, m))]
    for r in range(0, d, 2):
        s0 = int(rng.integers(0, T.size - m + 1))
        w = T[s0:s0 + m]
        if np.isin(w, A).all():
            P[r] = w
    P[-1] = P[0]
    P[d // 2] = A[0]
    return P


@pytest.mark.parametrize("m", [1, 2, 5, 8, 9, 12, 16, 17, 24, 31, 32, 48, 65])
@pytest.mark.parametrize("alphabet", [b"ACGT", b"acgt", b"AB", b"ACDEFGHIKLMNPQRSTVWY"])
def test_one_length(alphabet, m):
    rng = np.random.default_rng(900 + m + len(alphabet))
    for d in (3, 60, 2500 if m == 16 else 700):  # 2500: built on a thread of its own
        T = _text(rng, alphabet, 20011)
        P = _rows(rng, T, alphabet, d, m)
        want = oracle.dictionary(T, P, threads=THREADS)
        for h in (pm.pm_ac_compile(P, HOST), pm.pm_wm_compile(P, min(2, m), HOST), pm.pm_pfac_compile(P, HOST)):
            try:
                try:
                    occ, cnt = pm.pm_selfcheck_gram_walk(h, T)
                except pm.PmError as e:
                    assert e.code == pm.PM_EINVAL  # no gram fits, or too many matches
                    assert m < 3 or len(alphabet) ** min(m, 16) < 80 * d
                    continue
                assert np.array_equal(occ, want[0]) and np.array_equal(cnt, want[1]), (alphabet, m, d)
            finally:
                pm.pm_set_free(h)


@pytest.mark.parametrize("lo,hi", [(1, 6), (4, 9), (8, 16), (16, 40), (20, 65)])
@pytest.mark.parametrize("alphabet", [b"ACGT", b"ACGTN", b"ab"])
def test_mixed_lengths(alphabet, lo, hi):
    rng = np.random.default_rng(77 + lo + len(alphabet))
    A = np.frombuffer(alphabet, np.uint8)
    T = _text(rng, alphabet, 15013)
    P = []
    for r in range(300):
        L = int(rng.integers(lo, hi + 1))
        s0 = int(rng.integers(0, T.size - L + 1))
        P.append(bytes(T[s0:s0 + L]) if r % 2 else bytes(A[rng.integers(0, A.size, L)]))
    P += [P[0], P[1][:lo], bytes([A[0]]) * lo, bytes([A[0]]) * hi]
    want = oracle.dictionary_var(T, P, threads=THREADS)
    for h in (pm.pm_acv_compile(P, HOST), pm.pm_wmv_compile(P, min(2, lo), HOST)):
        try:
            try:
                occ, cnt = pm.pm_selfcheck_gram_walk(h, T)
            except pm.PmError as e:
                assert e.code == pm.PM_EINVAL and lo < 4
                continue
            assert np.array_equal(occ, want[0]) and np.array_equal(cnt, want[1])
        finally:
            pm.pm_set_free(h)


def test_large_set():
    rng = np.random.default_rng(3)
    T = _text(rng, b"ACGT", 60013)
    P = _rows(rng, T, b"ACGT", 17000, 32)
    want = oracle.dictionary(T, P, threads=THREADS)
    h = pm.pm_ac_compile(P, HOST)
    try:
        occ, cnt = pm.pm_selfcheck_gram_walk(h, T)
        assert np.array_equal(occ, want[0]) and np.array_equal(cnt, want[1])
    finally:
        pm.pm_set_free(h)


def test_text_edges():
    P = np.frombuffer(b"ACGTACGTACGTACGTACGTACGTACGTACGT", np.uint8).reshape(1, 32)
    h = pm.pm_ac_compile(P, HOST)
    try:
        for n in (0, 1, 31, 32, 33, 47, 48, 49, 95, 96):
            T = np.frombuffer(b"ACGT" * 24, np.uint8)[:n]
            want = oracle.dictionary(T, P, threads=1)
            occ, cnt = pm.pm_selfcheck_gram_walk(h, T)
            assert np.array_equal(occ, want[0]) and np.array_equal(cnt, want[1])
    finally:
        pm.pm_set_free(h)


@pytest.mark.parametrize("pin", ["placement", "smem_table_bytes", "warps_per_cta", "ctas_per_sm", "counters",
                                 "ids_place", "stride"])
def test_pinned_plans_keep_the_automaton(pin):
    h = pm.pm_ac_compile([b"ACGTACGTACGT"], dict(HOST, **{pin: 2}))
    try:
        with pytest.raises(pm.PmError) as e:
            pm.pm_selfcheck_gram_walk(h, np.frombuffer(b"ACGT" * 8, np.uint8))
        assert e.value.code == pm.PM_EINVAL
    finally:
        pm.pm_set_free(h)


def test_huge_groups_keep_the_automaton():
    """A tile's keys are added up in 32 bits: 2^18 equal patterns have no gram plan."""
    P = np.tile(np.frombuffer(b"ACGTACGTAC", np.uint8), (1 << 18, 1))
    for d, ok in ((1 << 18, False), ((1 << 18) - 1, True)):
        h = pm.pm_wm_compile(P[:d], 2, HOST)
        try:
            if ok:
                occ, _ = pm.pm_selfcheck_gram_walk(h, np.frombuffer(b"TACGTACGTACC", np.uint8))
                assert occ.size == d
            else:
                with pytest.raises(pm.PmError):
                    pm.pm_selfcheck_gram_walk(h, np.frombuffer(b"TACGTACGTACC", np.uint8))
        finally:
            pm.pm_set_free(h)


def test_repetitive_sets_keep_the_automaton():
    """A gram with more than 256 entries: an Aho-Corasick set keeps its table."""
    rng = np.random.default_rng(8)
    P = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, (400, 32))]
    P[:, :24] = ord("A")
    T = np.full(3000, ord("A"), np.uint8)
    T[1000:1032] = P[7]
    want = oracle.dictionary(T, P, threads=1)
    h = pm.pm_ac_compile(P, HOST)
    try:
        with pytest.raises(pm.PmError):
            pm.pm_selfcheck_gram_walk(h, T)
        assert np.array_equal(pm.pm_selfcheck_host_walk(h, T)[0], want[0])
    finally:
        pm.pm_set_free(h)
    h = pm.pm_wm_compile(P, 2, HOST)
    try:
        assert np.array_equal(pm.pm_selfcheck_gram_walk(h, T)[0], want[0])
    finally:
        pm.pm_set_free(h)
