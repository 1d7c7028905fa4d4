"""pkr_plan_bytes counts the third population array of per-step-checked binary64
runs exactly for the problems that may allocate it: the default geometry, at
most two 32-site tiles per SM, tau_lb != 1."""
import ctypes

import pytest


@pytest.fixture(scope="module")
def pk():
    from paper_1504_05869_gb300 import build
    build.build()
    import paper_1504_05869_gb300 as pkg
    pkg._pkr.load()
    return pkg


@pytest.mark.parametrize("shape,tau,variant,precision,arrays", [
    ((64, 64), 1.5, -1, "fp64", 3), ((64, 152), 1.5, -1, "fp64", 3),
    ((64, 153), 1.5, -1, "fp64", 2), ((64, 64), 1.5, 2, "fp64", 2),
    ((64, 64), 1.0, -1, "fp64", 2), ((64, 64), 1.5, -1, "fx64", 2),
])
def test_third_array_of_resident_runs(pk, shape, tau, variant, precision, arrays):
    p = pk.problem("D2Q169", shape, 7, tau_lb=tau, variant=variant, precision=precision)
    b = ctypes.c_size_t()
    assert pk._pkr.pkr_plan_bytes(ctypes.byref(p), ctypes.byref(b)) == 0
    V = shape[0] * shape[1]
    rest = b.value - arrays * (169 * V * 8 + 16)
    assert 0 < rest < 2 * V * 8 + 5 * 152 * 32 * 8      # S, Phi and the scratch
