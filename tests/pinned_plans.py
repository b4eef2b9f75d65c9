"""Automatic launch plans take the gram scan where the set has it. These
fixtures compile such sets with one CTA per SM pinned, which is what the
planners take anyway and keeps the method's own scan, so that a module can run
the tests of another one on the kernels they were written for."""
import pytest

from paper_1407_2889_gb300 import pmscan as pm

PINNED = {"ctas_per_sm": 1}
_COMPILERS = ("ac", "pfac", "wm", "acv", "wmv")


@pytest.fixture(scope="module", autouse=True)
def own_scans():
    with pytest.MonkeyPatch.context() as mp:
        for name in _COMPILERS:
            mp.setattr(pm.PatternSet, name, staticmethod(_pinned(name)))
        yield


def _pinned(name):
    make = getattr(pm.PatternSet, name)
    nargs = 2 if name in ("wm", "wmv") else 1   # patterns, and the block size

    def compile_(*args):
        params = args[nargs] if len(args) > nargs else None
        s = make(*args[:nargs], dict(PINNED) if not params else params)
        assert params or s.scan_kind() == pm.PM_SCAN_METHOD
        return s

    return compile_
