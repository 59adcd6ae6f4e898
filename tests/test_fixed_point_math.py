"""The fp64 kernel's fixed-point exponential and logarithms and its reciprocal against extended precision
(numpy's longdouble: 64 bits of mantissa or more), at the errors that the kernel counts on:

* 2^x: 0.51 ulp, at the edges of both tables (fractions that are multiples of 2^-10 and 2^-20, and their
  neighbours) and at the ends of its range;
* exp, from a longer argument of the same routine for |x| < 700: 1 ulp, around powers of 2 too;
* log2 in units of 2^-58: 6 units, at the edges of its 256 intervals; in units of 2^-52 over the whole
  range of fp64, one unit (truncation) more;
* reciprocal: 2 ulp.

And the mixed kernel's double-float ln for |ln x| < 16: the roundings of low parts of at most 2^-21, six
of them, 6 x 2^-46.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L = np.longdouble


def _math(op, x, fn="diag_fixed_math"):
    import torch
    from paper_2506_02602_gb300 import build, chem
    build.build()
    return getattr(chem, fn)(op, torch.tensor(x, dtype=torch.float64, device="cuda")).cpu().numpy()


def _ulps(got, ref):
    return np.abs(got.astype(L) - ref) / np.spacing(np.abs(ref.astype(np.float64))).astype(L)


def test_exp2():
    rng = np.random.default_rng(21)
    y = [rng.uniform(-1019.0, 1019.0, 200000), rng.uniform(-1.0, 1.0, 100000), [0.0, 1019.9, -1019.9, -2.0**-52, 2.0**-52]]
    for step in (2.0**-10, 2.0**-20):
        edge = rng.integers(-900, 900, 4000) + rng.integers(0, 1024, 4000) * step
        y += [edge, edge - 2.0**-42, edge + 2.0**-42, -edge]
    x = np.round(np.concatenate(y) * 2.0**52) / 2.0**52
    got = _math(0, x)
    err = _ulps(got, np.exp2(x.astype(L)))
    print(f"\n2^x: {float(err.max()):.4f} ulp")
    assert err.max() <= 0.51
    assert got[300000] == 1.0


def test_exp():
    rng = np.random.default_rng(22)
    x = np.concatenate([rng.uniform(-700.0, 700.0, 200000), rng.uniform(-1.0, 1.0, 100000),
                        rng.uniform(-1.0, 1.0, 1000) * 2.0 ** -rng.integers(1, 70, 1000),
                        [700.0 - 1e-10, -700.0 + 1e-10, 0.0, 5e-324]])
    k = np.arange(-1009, 1010) * np.log(2.0)  # powers of 2, from either side
    x = np.concatenate([x, k, np.nextafter(k, -1e9), np.nextafter(k, 1e9)])
    err = _ulps(_math(0, x, "diag_math"), np.exp(x.astype(L)))
    print(f"\nexp: {float(err.max()):.4f} ulp")
    assert err.max() <= 1.0
    edge = np.array([700.0, -700.0, 700.1, -700.1, 705.0, -705.0])
    assert _ulps(_math(0, edge, "diag_math"), np.exp(edge.astype(L))).max() <= 2.0


def _log2_points(rng, lo, hi, n):
    f = np.concatenate([rng.uniform(1.0, 2.0, n), 1.0 + np.arange(256) / 256.0,
                        np.nextafter(1.0 + np.arange(1, 257) / 256.0, 0.0), [1.0, np.nextafter(2.0, 0.0)]])
    x = f * 2.0 ** rng.integers(lo, hi, f.size)
    return np.concatenate([x, f])


def test_log2():
    rng = np.random.default_rng(23)
    x = _log2_points(rng, -31, 31, 100000)
    got = _math(1, x).view(np.int64)
    err = np.abs(got.astype(L) - np.log2(x.astype(L)) * L(2) ** 58)
    print(f"\nlog2: {float(err.max()):.2f} units of 2^-58")
    assert err.max() <= 6.0
    x = np.concatenate([_log2_points(rng, -1022, 1023, 100000), [2.0**-1022, np.finfo(float).max]])
    err = _math(2, x).view(np.int64).astype(L) - np.log2(x.astype(L)) * L(2) ** 52
    assert err.max() <= 6.0 / 64 and err.min() >= -1.0 - 6.0 / 64


def test_reciprocal():
    rng = np.random.default_rng(24)
    x = np.concatenate([np.exp(rng.uniform(-690, 690, 200000)), rng.uniform(128.0, 8192.0, 100000),
                        2.0 ** np.arange(-1020.0, 1021.0), np.nextafter(2.0 ** np.arange(-1000.0, 1000.0), 0.0)])
    x = np.concatenate([x, -x])
    err = _ulps(_math(3, x), 1 / x.astype(L))
    print(f"\nreciprocal: {float(err.max()):.3f} ulp")
    assert err.max() <= 2.0


def test_double_float_log():
    rng = np.random.default_rng(25)
    j = 1.0 + (np.arange(65) - 0.5) / 64.0  # the table's interval edges
    f = np.concatenate([j[1:], np.nextafter(j[1:].astype(np.float32), np.float32(0)).astype(np.float64),
                        1.0 + np.arange(64) / 64.0])
    x = np.concatenate([rng.uniform(100.0, 9000.0, 200000), np.exp(rng.uniform(-15.9, 15.9, 100000)),
                        *(f * 2.0**e for e in (-20, -1, 0, 8, 12)), 1.0 + np.linspace(-1e-6, 1e-6, 2001)])
    h = x.astype(np.float32).astype(np.float64)
    x = h + (x - h).astype(np.float32)  # a pair
    err = np.abs(_math(4, x).astype(L) - np.log(x.astype(L)))
    print(f"\nln in double-float: {float(err.max()):.3g}")
    assert err.max() <= 6 * 2.0**-46
