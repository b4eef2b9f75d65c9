"""Sets whose grams are poor keep their method's own scan: patterns that share
long runs of one letter, dense sets that hold most m-grams, mixed lengths with
many patterns of a few characters. And ordinary sets beside them take grams."""
import numpy as np
import pytest

import oracle
from paper_1407_2889_gb300 import pmscan as pm

HOST = {"host_only": 1}


def _rows(alphabet, d, m, seed=1):
    A = np.frombuffer(alphabet, np.uint8)
    return A[np.random.default_rng(seed).integers(0, A.size, (d, m))]


def _mixed(alphabet, d, lo, hi, seed=2):
    rng = np.random.default_rng(seed)
    return [bytes(r[:rng.integers(lo, hi + 1)]) for r in _rows(alphabet, d, hi, seed)]


def _kind(h):
    try:
        return pm.pm_set_scan_kind(h)
    finally:
        pm.pm_set_free(h)


@pytest.mark.parametrize("alphabet", [b"ACGT", b"ACDEFGHIKLMNPQRSTVWY"])
def test_repetitive_sets(alphabet):
    P = _rows(alphabet, 900, 32)
    V = [bytes(r) + bytes(r[:k % 16]) for k, r in enumerate(P)]
    plain = [pm.pm_ac_compile(P, HOST), pm.pm_pfac_compile(P, HOST), pm.pm_wm_compile(P, 2, HOST),
             pm.pm_wm_compile(P, 4, HOST), pm.pm_acv_compile(V, HOST)]
    assert [_kind(h) for h in plain] == [pm.PM_SCAN_GRAMS] * 5
    P[:400, :24] = ord("A")     # 3,600 entries under a gram of 16 A
    V = [bytes(r) + bytes(r[:k % 16]) for k, r in enumerate(P)]
    T = np.full(2000, ord("A"), np.uint8)
    T[900:932] = P[7]
    want, want_var = oracle.dictionary(T, P, threads=1), oracle.dictionary_var(T, V, threads=1)
    for h, w in ((pm.pm_pfac_compile(P, HOST), want), (pm.pm_acv_compile(V, HOST), want_var)):
        try:
            with pytest.raises(pm.PmError):
                pm.pm_selfcheck_gram_walk(h, T)
            assert np.array_equal(pm.pm_selfcheck_host_walk(h, T)[0], w[0])
        finally:
            assert _kind(h) == pm.PM_SCAN_METHOD
    for B in (2, 4):            # the tables stay for the host walk
        h = pm.pm_wm_compile(P, B, HOST)
        assert np.array_equal(pm.pm_selfcheck_gram_walk(h, T)[0], want[0])
        assert _kind(h) == pm.PM_SCAN_METHOD


def test_limits_by_method():
    """9 f entries under a gram of 16 A, and a few that share its bucket."""
    def kinds(f):
        P = _rows(b"ACGT", 2000, 32)
        P[:f, :25] = np.frombuffer(b"A" * 24 + b"C", np.uint8)   # 9 grams of 16 A each
        return [_kind(pm.pm_ac_compile(P, HOST)), _kind(pm.pm_pfac_compile(P, HOST)),
                _kind(pm.pm_wm_compile(P, 2, HOST)), _kind(pm.pm_wm_compile(P, 4, HOST))]
    G, M = pm.PM_SCAN_GRAMS, pm.PM_SCAN_METHOD
    assert kinds(27) == [G, G, G, G]
    assert kinds(30) == [M, G, G, M]
    assert kinds(111) == [M, G, G, M]
    assert kinds(115) == [M, M, M, M]


def test_byte_hash_wu_manber_that_compares_every_window():
    """Mixed lengths past 32 and blocks that name hundreds of patterns: grams
    win however long the list, until a tile's key sum needs more than 32 bits."""
    P = _rows(b"ACGT", 3000, 48)
    P[:, :24] = ord("A")
    V = [bytes(r[:32 + k % 17]) for k, r in enumerate(P)]
    assert _kind(pm.pm_wmv_compile(V, 2, HOST)) == pm.PM_SCAN_GRAMS
    assert _kind(pm.pm_wmv_compile(V, 4, HOST)) == pm.PM_SCAN_METHOD
    V = [b"ACGTACGTAC"] * (1 << 18) + [b"C" * 40]
    assert _kind(pm.pm_wmv_compile(V, 2, HOST)) == pm.PM_SCAN_METHOD


@pytest.mark.parametrize("d,m,dense", [(300, 5, True), (3000, 6, True), (3000, 5, False), (300, 4, False)])
def test_dense_sets_of_most_grams(d, m, dense):
    P = _rows(b"ACGT", d, m)
    for make in (pm.pm_ac_compile, pm.pm_pfac_compile):
        assert _kind(make(P, HOST)) == (pm.PM_SCAN_DENSE if dense else pm.PM_SCAN_METHOD)
    assert _kind(pm.pm_wm_compile(P, 2, HOST)) == pm.PM_SCAN_DENSE   # never faster


@pytest.mark.parametrize("lo,hi,d,kind", [
    (6, 20, 20000, pm.PM_SCAN_GRAMS), (4, 40, 1000, pm.PM_SCAN_GRAMS), (4, 40, 20000, pm.PM_SCAN_METHOD),
    (3, 65, 3000, pm.PM_SCAN_METHOD), (3, 20, 60000, pm.PM_SCAN_GRAMS)])
def test_mixed_lengths_with_many_short_patterns(lo, hi, d, kind):
    V = _mixed(b"ACGT", d, lo, hi)
    assert _kind(pm.pm_acv_compile(V, HOST)) == kind
    if d <= 3000:
        assert _kind(pm.pm_wmv_compile(V, 2, HOST)) == pm.PM_SCAN_GRAMS


@pytest.mark.parametrize("lo,hi,d,kind", [(10, 20, 1000, pm.PM_SCAN_METHOD), (16, 24, 1000, pm.PM_SCAN_GRAMS),
                                          (8, 20, 2000, pm.PM_SCAN_GRAMS)])
def test_mixed_lengths_over_two_letters(lo, hi, d, kind):
    """A small automaton and few matches beat grams that half of all windows pass."""
    assert _kind(pm.pm_acv_compile(_mixed(b"AC", d, lo, hi), HOST)) == kind
