"""Accuracy of the Voigt kernel's slow-zone forms (rox_faddeeva.cuh, rox_core_tables.h), compiled
for the host, against scipy.special.wofz over each line's slow zone: y from 1e-9 to 22, both sides
of every interval of the coefficient tables.

Tolerance: the rational interpolants are within 5e-7 of Re w (against Re w, Gaussian part included);
Horner's rule with positive denominators adds at most 17 roundings of 6e-8, and for y < 0.1 the
exponential of an argument of up to 61 rounded twice adds 61 x 2 x 6e-8 x ln 2 / 2 = 2.5e-6 where it
dominates. Hence 4e-6."""
import ctypes

import numpy as np
import pytest
from scipy.special import wofz

EDGES = (0.1, 0.2, 0.4, 0.55, 0.75, 1.0, 1.5, 2.0, 2.5, 3.5, 5.0, 7.5, 11.5)


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    lib = ctypes.CDLL(__graft_entry__._build_module().build_host_lib())
    lib.rox_host_core_zone.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int64]
    lib.rox_host_far_r2.argtypes = [ctypes.c_float]
    lib.rox_host_far_r2.restype = ctypes.c_float
    return lib


def _ys(lo, hi):
    return np.exp(np.linspace(np.log(lo), np.log(hi), 40)).astype(np.float32)


@pytest.mark.parametrize("lo,hi", [(1e-9, 1e-3), (1e-3, 0.0999999)] + list(zip(EDGES, EDGES[1:] + (21.99,))))
def test_zone_form(lib, lo, hi):
    worst = 0.0
    for y in _ys(lo, hi):
        r2 = lib.rox_host_far_r2(float(y))
        if r2 <= float(y) ** 2:
            continue
        x = np.linspace(0.0, np.sqrt(r2 - float(y) ** 2) * 1.0002, 1500).astype(np.float32)
        out, yy = np.empty_like(x), np.full_like(x, y)
        lib.rox_host_core_zone(x.ctypes.data, yy.ctypes.data, out.ctypes.data, x.size)
        ref = wofz(x.astype(np.float64) + 1j * float(y)).real
        m = ref > 1e-15            # below 1e-15 of the line peak nothing can reach the tolerance
        worst = max(worst, float((np.abs(out - ref)[m] / ref[m]).max()))
        assert np.all(np.abs(out - ref)[~m] < 2e-15)
    assert worst < 4e-6, worst
