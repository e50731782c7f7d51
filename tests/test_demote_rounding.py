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


def _transform_f32(x):
    """The kernel's order: H_16 on every block of 16 dims, then butterflies over the blocks, all in fp32."""
    x, d = x.astype(F).copy(), x.shape[-1]
    for strides in ([1, 2, 4, 8], [16 << i for i in range(d.bit_length() - 5)]):
        for h in strides:
            v = x.reshape(*x.shape[:-1], -1, 2, h)
            x = np.stack([v[..., 0, :] + v[..., 1, :], v[..., 0, :] - v[..., 1, :]], -2).reshape(x.shape)
            assert x.dtype == F
    return x


def _transform_units(x):
    """The same in units of 2^-9, exactly."""
    x, d = np.rint(x * 512.0).astype(np.int64), x.shape[-1]
    for h in [1 << i for i in range(d.bit_length() - 1)]:
        v = x.reshape(*x.shape[:-1], -1, 2, h)
        x = np.stack([v[..., 0, :] + v[..., 1, :], v[..., 0, :] - v[..., 1, :]], -2).reshape(x.shape)
    return x


def _gate():
    import os
    import re

    from conftest import ROOT
    with open(os.path.join(ROOT, "paper_2608_23834_b200", "csrc", "demote_warp.cuh")) as f:
        return float(re.search(r"kExactNorm2 = ([0-9.]+)f;", f.read()).group(1))


def test_transform_is_exact_below_the_norm_gate_and_not_far_above():
    """Vectors whose squared norm lies just below the kernel's gate, among them those that reach the largest sums: a
    row of the transform's own signs scaled to the gate (one coordinate of 2^24 units), with the odd last bits that
    small values bring.  Beyond the gate the fp32 sums do round, which is why there is one."""
    gate, v, rng = _gate(), _e4m3_values(), np.random.default_rng(1)
    assert gate == 2.0 ** 22
    rows = []
    for d in (128, 256):
        signs = np.where(rng.random((64, d)) < 0.5, -1.0, 1.0)
        for top in (96.0, 112.0, 120.0, 128.0, 144.0, 176.0, 448.0):
            x = top * np.ones((64, d)) * np.where(np.arange(64)[:, None] % 2, signs, 1.0)
            small = rng.random((64, d)) < rng.uniform(0, 0.5, (64, 1))
            x = np.where(small, rng.choice(v[np.abs(v) < 0.1], (64, d)), x)
            x[(x ** 2).sum(-1) >= gate] = 0.0
            rows.append(x)
        x = rng.choice(v, (4096, d))
        rows.append(x[(x ** 2).sum(-1) < gate])
    largest = 0
    for x in rows:
        want = _transform_units(x)
        assert np.array_equal(_transform_f32(x).astype(np.float64) * 512.0, want.astype(np.float64))
        largest = max(largest, int(np.abs(want).max()))
    assert largest > 2 ** 23                                          # the cases do come near the 2^24 of the argument
    x = np.full((1, 256), 448.0)
    x[0, 3] = 2.0 ** -9                                               # an odd sum of 26 bits
    assert not np.array_equal(_transform_f32(x).astype(np.float64) * 512.0, _transform_units(x).astype(np.float64))
