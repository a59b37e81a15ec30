"""The small projected solver called directly (mof::launch_small_solve), for calls that the
public entry points do not make at will."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2501_12497_gb300 import api

P, I, D = ctypes.c_void_p, ctypes.c_int, ctypes.c_double


class SmallArgs(ctypes.Structure):  # csrc/solver.cuh
    _fields_ = ([(n, P) for n in ("GA", "GL", "g", "bb", "K", "active")] + [(n, I) for n in ("ld", "B", "rule")] +
                [("target2", D), ("lam_fixed", D)] +
                [(n, P) for n in ("lam", "z", "flag", "err", "Mg", "Linv", "nL", "proj", "Y", "Yd", "Yh", "Yrho", "nY")])


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    return api.load()


def _launch(lib, args):
    fn = lib["_ZN3mof18launch_small_solveERKNS_9SmallArgsEP11CUstream_st"]
    fn.argtypes, fn.restype = [ctypes.POINTER(SmallArgs), P], I
    return fn(ctypes.byref(args), None)
