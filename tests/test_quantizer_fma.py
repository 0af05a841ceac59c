"""The flush kernel's code computation, restated in numpy: p = (x - z) * RN(1 / s) rounded by adding 1.5 * 2^23, its distance d
from that integer, the division only within 4e-6 of one half and not for exact ties, or where p is NaN.  Equal to the clamped
round-half-even of the IEEE quotient for every input tried.  (Products are exact in float64, so its one rounding stands for the
FMA's.)"""
import numpy as np

MARGIN = np.float32(0.5) - np.float32(4e-6)


def bf16_down(x):
    return (np.asarray(x, np.float32).view(np.uint32) & np.uint32(0xFFFF0000)).view(np.float32)


def exact_codes(t, s, max_code):
    with np.errstate(all="ignore"):
        y = np.rint((t / s).astype(np.float32))
    return np.where(np.isnan(y), 0, np.clip(y, 0, max_code)).astype(np.int64)


def kernel_codes(t, s, max_code):
    with np.errstate(all="ignore"):
        r = (np.float32(1) / s).astype(np.float32)
        r = np.where(np.isinf(r), np.float32(np.nan), r)
        p = t.astype(np.float64) * r.astype(np.float64)
        c = np.rint(p)
        d = (p - c).astype(np.float32)
        ok = np.abs(d) <= MARGIN
        tie = (c + np.copysign(0.5, d.astype(np.float64))) * s.astype(np.float64) - t.astype(np.float64) == 0
        even = np.where(c % 2 == 0, c, np.where(d > 0, c + 1, c - 1))
    code = np.where(ok, c, np.where(tie, even, exact_codes(t, s, max_code)))
    return code.astype(np.int64) & 15, ok


def test_random_groups_over_all_scales():
    rng = np.random.default_rng(7)
    for max_code in (3, 15):
        e = rng.integers(-133, 124, 200000)               # subnormal scales among them
        s = bf16_down(np.ldexp(rng.uniform(1, 2, e.size), e))
        s = s[s > 0]
        t = (rng.uniform(0, max_code, s.size) * s).astype(np.float32)
        t[::7] = 0.0
        t[1::7] = (max_code * s.astype(np.float64)).astype(np.float32)[1::7]
        got, ok = kernel_codes(t, s, max_code)
        assert np.array_equal(got, exact_codes(t, s, max_code))
        assert not ok[s <= np.float32(2.0 ** -128)].any() and ok[s >= np.float32(2.0 ** -126)].mean() > 0.99


def test_on_and_beside_the_ties():
    rng = np.random.default_rng(11)
    s = bf16_down(np.exp(rng.uniform(-60, 60, 20000)).astype(np.float32))
    for max_code in (3, 15):
        for k in range(max_code):
            tie = ((k + 0.5) * s.astype(np.float64)).astype(np.float32)
            for ulps in range(-12, 13):
                t = (tie.view(np.int32) + ulps).view(np.float32)
                assert np.array_equal(kernel_codes(t, s, max_code)[0], exact_codes(t, s, max_code)), (max_code, k, ulps)


def test_elements_that_are_not_finite():
    s = np.array([1, 1, np.inf, np.inf, np.inf, 2.0 ** -130], np.float32)
    t = np.array([np.nan, 2, np.inf, 5, np.nan, np.nan], np.float32)
    assert kernel_codes(t, s, 3)[0].tolist() == exact_codes(t, s, 3).tolist() == [0, 2, 0, 0, 0, 0]
