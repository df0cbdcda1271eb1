"""The pair-of-floats form of the line strength (rox_strength_df.h), compiled for the host, against
the strength formula in 40 digits: its error bound, and that the rounding it calls certain is the
correctly rounded FP32 value.

Bound: the bound the code itself relies on (2^-35). By count of roundings: the third-order term of the
exponential's series is off by four FP32 roundings (2^-24 each) of 2^-15.6 of its argument, 2^-37.6, twice
where two stimulated-emission factors are divided; every other term is below 2^-44."""
import ctypes

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")

C2, C, T_REF = 1.4387768775039338, 2.99792458e10, 296.0


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    lib = ctypes.CDLL(__graft_entry__._build_module().build_host_lib())
    D, P = ctypes.c_double, ctypes.c_void_p
    lib.rox_host_strength_df.argtypes = [ctypes.c_int, D, D, D, D] + [P] * 9 + [ctypes.c_int64]
    return lib


def _run(lib, conv, T, q, nu0, a, g, el):
    hit = int(conv == 0)
    c2_dT = C2 * (1 / T - 1 / T_REF) if hit else C2 / T
    fac = q if hit else q / (8 * np.pi * C)
    n = nu0.size
    hi, lo, rd = (np.zeros(n, np.float32) for _ in range(3))
    ex, ok = np.zeros(n, np.int32), np.zeros(n, np.uint8)
    lib.rox_host_strength_df(hit, c2_dT, fac, C2 / T, C2 / T_REF, *(v.ctypes.data for v in (nu0, a, g, el, hi, lo, ex, rd, ok)),
                             n)
    return hi, lo, ex, rd, ok, c2_dT, fac


@pytest.mark.parametrize("conv", [0, 1])
@pytest.mark.parametrize("T", [20.0, 100.0, 296.0, 300.0, 1500.0, 8000.0])
def test_pair_strengths(lib, conv, T):
    rng = np.random.default_rng(int(T) + conv)
    n = 1500
    nu0 = np.exp(rng.uniform(np.log(1e-3), np.log(5e5), n))
    nu0[:400] = np.exp(rng.uniform(np.log(0.02 * T), np.log(2.0 * T), 400))   # stimulated emission near 1
    a = np.exp(rng.uniform(np.log(1e-30), np.log(1e3), n)).astype(np.float32)
    g = rng.integers(1, 300, n).astype(np.float32)
    el = rng.uniform(-10.0, 4e4, n).astype(np.float32) * rng.choice([1.0, 0.01], n).astype(np.float32)
    hi, lo, ex, rd, ok, c, fac = _run(lib, conv, T, 0.37, nu0, a, g, el)
    used = ex != np.iinfo(np.int32).min
    assert used[np.abs(el * c) < 600].mean() > 0.95
    worst, certain = 0.0, 0
    with mp.workdps(40):
        for i in np.flatnonzero(used):
            stim = -mp.expm1(-mp.mpf(C2 / T) * mp.mpf(nu0[i]))
            S = mp.mpf(float(a[i])) * mp.mpf(fac) * mp.exp(-mp.mpf(float(el[i])) * mp.mpf(c)) * stim
            if conv == 0:
                S /= -mp.expm1(-mp.mpf(C2 / T_REF) * mp.mpf(nu0[i]))
            else:
                S *= mp.mpf(float(g[i])) / mp.mpf(nu0[i]) ** 2
            got = mp.ldexp(mp.mpf(float(hi[i])) + mp.mpf(float(lo[i])), int(ex[i]))
            worst = max(worst, float(abs(got / S - 1)))
            if ok[i]:
                certain += 1
                ref = np.float32(float(S)) if S < 3.4e38 else np.float32(np.inf)
                assert rd[i] == ref, (i, rd[i], ref)
    print(f"PARITY strength pairs conv {conv} T {T}: max rel err {worst:.3e} = 2^{np.log2(worst):.1f}, certain {certain / used.sum():.4f}")
    assert worst < 2.0 ** -35


def test_declined_operands(lib):
    """Operands outside the pair form's range are left to the FP64 form."""
    nu0 = np.array([1e3, 1e3, 1e3, 1e3, -5.0, 0.0, 2e6, np.nan, 1e3, 1e3])
    a = np.array([0.0, -1e-20, np.inf, 1e-42, 1, 1, 1, 1, np.nan, 1], dtype=np.float32)
    el = np.array([10.0] * 9 + [np.nan], dtype=np.float32)
    ex = _run(lib, 0, 500.0, 1.0, nu0, a, np.ones(10, np.float32), el)[2]
    assert np.all(ex == np.iinfo(np.int32).min)
