"""Which roundings of the pair form (rox_strength_df.h) are called certain: nearly all of ordinary lines
(all but 2^-35 / 2^-25 of them and twice that, about one in 500, so 99% are asked for), none that could go
the other way within the form's error of 2^-35, and the right value in the subnormal range and below."""
import ctypes

import numpy as np
import pytest


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    lib = ctypes.CDLL(__graft_entry__._build_module().build_host_lib())
    D, P = ctypes.c_double, ctypes.c_void_p
    lib.rox_host_strength_df.argtypes = [ctypes.c_int, D, D, D, D] + [P] * 9 + [ctypes.c_int64]
    lib.rox_host_df_round.argtypes = [P] * 5 + [ctypes.c_int64]
    return lib


def _round(lib, h, l, e):
    h, l = np.asarray(h, np.float32), np.asarray(l, np.float32)
    e = np.asarray(np.broadcast_to(e, h.shape), np.int32).copy()
    out, ok = np.zeros(h.size, np.float32), np.zeros(h.size, np.uint8)
    lib.rox_host_df_round(*(v.ctypes.data for v in (h, l, e, out, ok)), h.size)
    return out, ok.astype(bool)


@pytest.mark.parametrize("conv", [0, 1])
@pytest.mark.parametrize("T", [296.0, 1000.0, 3000.0])
def test_ordinary_lines_are_certain(lib, conv, T):
    rng = np.random.default_rng(int(T) + conv)
    n = 200_000
    nu0 = rng.uniform(300.0, 30000.0, n)
    a = np.exp(rng.uniform(*np.log([1e-30, 1e-19] if conv == 0 else [1e-8, 1e2]), n)).astype(np.float32)
    g, el = rng.integers(1, 101, n).astype(np.float32), rng.exponential(5000.0, n).astype(np.float32)
    c2 = 1.4387768775039338
    hi, lo, rd = (np.zeros(n, np.float32) for _ in range(3))
    ex, ok = np.zeros(n, np.int32), np.zeros(n, np.uint8)
    lib.rox_host_strength_df(int(conv == 0), c2 * (1 / T - 1 / 296.0) if conv == 0 else c2 / T, 0.4, c2 / T, c2 / 296.0,
                             *(v.ctypes.data for v in (nu0, a, g, el, hi, lo, ex, rd, ok)), n)
    assert np.all(ex != np.iinfo(np.int32).min)
    S = np.ldexp(hi.astype(np.float64) + lo, ex)
    normal = (S > 1.2e-38) & (S < 3.4e38)
    assert normal.mean() > 0.9 and ok[normal].mean() >= 0.99, ok[normal].mean()
    assert np.array_equal(rd[ok == 1], S[ok == 1].astype(np.float32))


@pytest.mark.parametrize("e", [-100, -20, 0, 90])
def test_near_the_middle_of_two_floats(lib, e):
    """l at half an ulp of h less a little: certain from 2^-34 away on, declined within 2^-36. h even
    and odd, just above a power of two and just below the next; both signs of l."""
    for bits in (0x3f800001, 0x3f800002, 0x3fc00000, 0x3fc00001, 0x3fffffff):
        h = np.array(bits, np.uint32).view(np.float32)
        for sign in (1.0, -1.0):
            for away, certain in ((0.0, False), (2.0 ** -37, False), (2.0 ** -36, False), (2.0 ** -33, True),
                                  (2.0 ** -30, True)):
                l = np.float32(sign * (2.0 ** -24 - away * float(h)))
                out, ok = _round(lib, [h], [l], e)
                assert ok[0] == certain, (hex(bits), sign, away)
                if certain:
                    assert out[0] == np.float32(np.ldexp(float(h), e))


def test_subnormal_and_zero(lib):
    e = np.array([-127, -130, -140, -148, -149, -150, -151, -160, -180, -300])
    h = np.full(e.size, 1.375, np.float32)
    l = np.full(e.size, 3e-9, np.float32)
    out, ok = _round(lib, h, l, e)
    want = np.ldexp(1.375 + float(l[0]), e).astype(np.float32)
    assert ok.all() and np.array_equal(out, want)
    assert (want[:4] > 0).all() and want[-1] == 0.0
    # halfway between two subnormal numbers: 2.5 and 0.5 units of 2^-149
    out, ok = _round(lib, [1.25, 1.25, 1.0], [0.0, 1e-12, 0.0], [-148, -148, -150])
    assert not ok.any()
    # beyond the largest float, and near it
    out, ok = _round(lib, [1.5, 1.5], [0.0, 0.0], [128, 127])
    assert list(ok) == [False, True] and out[1] == np.float32(1.5 * 2.0 ** 127)
