"""The rounding arguments behind the warp-per-head Demote kernel, checked over their whole (finite) domain on the CPU:
FP8 values with scale 1 are multiples of 2^-9 below 512, so ranges, scales and quotients can be enumerated."""
import numpy as np

F = np.float32


def _e4m3_values():
    out = []
    for b in range(127):
        e, m = b >> 3, b & 7
        out.append((m / 8 * 2.0 ** -6) if e == 0 else (1 + m / 8) * 2.0 ** (e - 7))
    pos = np.array(out)
    return np.unique(np.concatenate([-pos, pos]))                    # 253 finite values


def test_division_by_seven_from_a_rounded_reciprocal():
    v = _e4m3_values()
    x = np.unique(v[:, None] - v[None, :])
    x = x[x >= 0].astype(F)
    y = F(1.0 / 7.0)
    q = (x * y).astype(F)
    r = (x.astype(np.float64) - 7.0 * q.astype(np.float64)).astype(F)          # exact, as in an FMA
    got = (q.astype(np.float64) + r.astype(np.float64) * np.float64(y)).astype(F)
    want = (x / F(7.0)).astype(F)
    assert np.array_equal(got, want)


def test_value_code_from_an_approximate_quotient():
    """rint(RN(num / scale)) for every minimum, maximum and value between them, with the reciprocal a unit in
    the last place off (the bound of rcp.approx)."""
    v = _e4m3_values().astype(F)
    for mn in v:
        top = v[v >= mn]
        sc = ((top - mn) / F(7.0)).astype(np.float16).astype(F)               # one scale per maximum
        num = (top - mn).astype(F)
        ok = sc != 0
        n, s = np.meshgrid(num, sc[ok])
        inside = n <= np.repeat((top - mn)[ok][:, None], len(num), 1)
        n, s = n[inside], s[inside]
        want = np.clip(np.rint((n / s).astype(F)), 0, 7)
        for ulps in (-1, 0, 1):
            y = ((F(1.0) / s) * F(1 + ulps * 2.0 ** -23)).astype(F)
            snapped = (n.astype(np.float64) * y.astype(np.float64) + 40.0).astype(F)
            r = (snapped.astype(np.float64) + (12582912.0 - 40.0)).astype(F)
            assert np.array_equal(r.view(np.uint32) - np.uint32(0x4B400000), want.astype(np.uint32)), (mn, ulps)


def test_transform_sums_of_small_keys_are_exact_in_fp32():
    """|x|^2 < 4096 with d <= 256 bounds every signed partial sum by sqrt(256 * 4096) = 1024; in units of 2^-9 that is
    2^19, and the products with +-512 are integers of that size: far inside 24 bits."""
    assert np.sqrt(256 * 4096.0) * 2 ** 9 <= 2 ** 19
