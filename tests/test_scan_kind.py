"""pm_set_scan_kind without a GPU: the scan that a set's tables are planned for."""
import ctypes

import numpy as np
import pytest

from paper_1407_2889_gb300 import pmscan as pm

HOST = {"host_only": 1}


def _rows(d, m, alphabet=b"ACGT"):
    A = np.frombuffer(alphabet, np.uint8)
    return A[np.random.default_rng(d + m).integers(0, A.size, (d, m))]


@pytest.mark.parametrize("make,kind", [
    (lambda: pm.pm_ac_compile(_rows(2000, 8), HOST), pm.PM_SCAN_DENSE),
    (lambda: pm.pm_pfac_compile(_rows(2000, 8), HOST), pm.PM_SCAN_DENSE),
    (lambda: pm.pm_ac_compile(_rows(2000, 16), HOST), pm.PM_SCAN_GRAMS),
    (lambda: pm.pm_wm_compile(_rows(2000, 16), 2, HOST), pm.PM_SCAN_GRAMS),
    (lambda: pm.pm_acv_compile([bytes(r[:8 + k % 9]) for k, r in enumerate(_rows(300, 16))], HOST), pm.PM_SCAN_GRAMS),
    (lambda: pm.pm_ac_compile(_rows(2000, 16), dict(HOST, warps_per_cta=12)), pm.PM_SCAN_METHOD),
    (lambda: pm.pm_wm_compile(_rows(2000, 16), 2, dict(HOST, warps_per_cta=12)), pm.PM_SCAN_METHOD),
    (lambda: pm.pm_ac_compile(_rows(200, 3, b"ACDEFGHIKLMNPQRSTVWY"), HOST), pm.PM_SCAN_METHOD),
])
def test_kind(make, kind):
    h = make()
    try:
        assert pm.pm_set_scan_kind(h) == kind
    finally:
        pm.pm_set_free(h)


def test_null():
    assert pm.lib().pm_set_scan_kind(ctypes.c_void_p(0)) == -1
