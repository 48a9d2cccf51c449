"""The integer forms of the FP64 kernel functions (csrc/fixed64.cuh), compiled
for the host, against extended precision (numpy longdouble, 64 or 113 bits).

Bound: the fixed-point value carries an error below 2^-57 before the one
rounding to 53 bits (2^-53 at most), so 1.2e-16 relative; exp(-t) adds the
absolute error of t (64-bit fraction of t's own size, t 2^-58) to that."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2012_06925_gb300", "csrc")
SRC = r"""
#include "fixed64.cuh"
using namespace bldtt::fixed64;
extern "C" void inv(const double* d, long n, double* o) {
  for (long i = 0; i < n; ++i) o[i] = inv_r(d[3 * i], d[3 * i + 1], d[3 * i + 2]);
}
extern "C" void scr(const double* d, long n, double kappa, double* o) {
  const Screen k = make_screen(kappa);
  for (long i = 0; i < n; ++i) o[i] = screened_inv_r(d[3 * i], d[3 * i + 1], d[3 * i + 2], k);
}
extern "C" void reg(const double* d, long n, double kappa, double* o) {
  for (long i = 0; i < n; ++i) o[i] = inv_sqrt_r2_kappa2(d[3 * i], d[3 * i + 1], d[3 * i + 2], kappa);
}
extern "C" void fix(const double* xy, long n, double kd, double kappa, double* o) {
  const int k = (int)kd;
  const Screen sc = make_screen(kappa);
  for (long i = 0; i < n; ++i) {
    const double *x = xy + 6 * i, *y = x + 3;
    const i64 a = to_fixed(x[0], k) - to_fixed(y[0], k), b = to_fixed(x[1], k) - to_fixed(y[1], k),
              c = to_fixed(x[2], k) - to_fixed(y[2], k);
    const uint32_t top = fixed_top(a, b, c);
    int E;
    if (top < kFixedTop) { o[i] = -1; continue; }
    const u64 S = sum_squares_fixed(a, b, c, top, k, &E);
    o[i] = kappa < 0 ? inv_r_of(S, E) : screened_inv_r_of(S, E, sc);
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("fixed64")
    (d / "f.cpp").write_text(SRC)
    so = str(d / "f.so")
    subprocess.run([gxx, "-O2", "-shared", "-fPIC", "-I", CSRC, str(d / "f.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


def call(lib, name, d, *args):
    d = np.ascontiguousarray(d, dtype=np.float64)
    out = np.empty(len(d))
    p = ctypes.POINTER(ctypes.c_double)
    getattr(lib, name)(d.ctypes.data_as(p), ctypes.c_long(len(d)), *[ctypes.c_double(a) for a in args],
                       out.ctypes.data_as(p))
    return out


def vectors(kind, n=20000):
    rng = np.random.default_rng(["plain", "mixed", "scaled", "ulps"].index(kind))
    d = rng.uniform(-1, 1, (n, 3))
    if kind == "mixed":                       # components of very different sizes, zeros among them
        d *= 2.0 ** -rng.integers(0, 70, (n, 3))
        d[::7, 2] = 0.0
        d[::11, 1] = -0.0
    elif kind == "scaled":                    # all sizes at which r^2 is a normal number
        d *= 2.0 ** rng.integers(-500, 500, (n, 1))
    elif kind == "ulps":                      # powers of two and their neighbours
        d = np.sign(d) * np.where(rng.random((n, 3)) < 0.5, 1.0, np.nextafter(1.0, 2.0 * (rng.random((n, 3)) < 0.5)))
        d *= 2.0 ** rng.integers(-3, 4, (n, 3))
    return d


def radius(d):
    x = d.astype(np.longdouble)
    return np.sqrt((x * x).sum(axis=1))


def worst(got, want):
    return float(np.max(np.abs(got.astype(np.longdouble) / want - 1)))


@pytest.mark.parametrize("kind", ["plain", "mixed", "scaled", "ulps"])
def test_inverse_distance(lib, kind):
    d = vectors(kind)
    assert worst(call(lib, "inv", d), 1 / radius(d)) <= 1.2e-16


@pytest.mark.parametrize("kind", ["plain", "mixed", "ulps"])
@pytest.mark.parametrize("kappa", [0.0, 1e-300, 1e-5, 0.5, 1.7, 30.0, 400.0])
def test_screened(lib, kind, kappa):
    d = vectors(kind)
    r = radius(d)
    want = np.exp(-np.longdouble(kappa) * r) / r
    got = call(lib, "scr", d, kappa)
    keep = want > 1e-300
    err = np.abs(got[keep].astype(np.longdouble) / want[keep] - 1)
    assert np.all(err <= 1.3e-16 + kappa * r[keep] * 1.45 * 2.0 ** -58)
    assert np.all(got[~keep] <= 1e-299) and np.all(got >= 0)


@pytest.mark.parametrize("kappa", [0.0, 1e-9, 0.005, 1.0, 1e6])
def test_regularized(lib, kappa):
    d = vectors("mixed")
    r = radius(d)
    assert worst(call(lib, "reg", d, kappa), 1 / np.sqrt(r * r + np.longdouble(kappa) ** 2)) <= 1.2e-16


def test_ends_of_the_range(lib):
    """Where FP64's r^2 is 0 or infinite a pair contributes nothing, as it did."""
    d = np.array([[0, 0, 0], [-0.0, 0, 0], [1e-170, 0, 0], [5e-324, 0, 1e-310], [1e200, 0, 0], [0, -1e300, 1e300]])
    for name, args in (("inv", ()), ("scr", (0.5,)), ("reg", (0.005,))):
        assert np.all(call(lib, name, d, *args) == 0.0), name
    one = np.array([[1.0, 0, 0], [0, -0.5, 0], [3.0, 0, 4.0], [2.0 ** -500, 0, 0]])
    assert np.array_equal(call(lib, "inv", one), [1.0, 2.0, 0.2, 2.0 ** 500])
    assert call(lib, "scr", [[1e4, 0, 0]], 1.0)[0] == 0.0       # exp(-1e4) is 0 in FP64 too


@pytest.mark.parametrize("shift,scale", [(0.0, 1.0), (1e6, 1.0), (-3e9, 2.0 ** -20), (0.0, 2.0 ** 400),
                                         (5e-150, 2.0 ** -480)])
@pytest.mark.parametrize("kappa", [-1.0, 0.0, 0.7])
def test_fixed_coordinates(lib, shift, scale, kappa):
    """Coordinates in units of 2^-62 of the extent (offsets wrap around): 1.2e-16 for the evaluation
    and 2^-56 sqrt(3) for the units of the closest pairs taken (1/64 of the extent)."""
    rng = np.random.default_rng(1)
    xy = rng.uniform(-1, 1, (20000, 6))
    xy[::3, 3:] = xy[::3, :3] + rng.uniform(-1, 1, (len(xy[::3]), 3)) * 2.0 ** -rng.integers(0, 9, (len(xy[::3]), 1))
    xy[::5, 2] = xy[::5, 5]
    xy[:2] = [[-1, -1, -1, 1, 1, 1], [1, -1, 1, -1, 1, -1]]
    xy = np.clip(xy, -1, 1) * scale + shift
    w = np.ptp(xy.reshape(-1, 3), axis=0).max()
    k = 61 - int(np.floor(np.log2(w)))
    a = np.ascontiguousarray(xy)
    out = np.empty(len(a))
    p = ctypes.POINTER(ctypes.c_double)
    lib.fix(a.ctypes.data_as(p), ctypes.c_long(len(a)), ctypes.c_double(k), ctypes.c_double(kappa / scale),
            out.ctypes.data_as(p))
    x = a.astype(np.longdouble)
    r = np.sqrt(((x[:, :3] - x[:, 3:]) ** 2).sum(axis=1))
    want = np.exp(-np.longdouble(max(kappa, 0) / scale) * r) / r
    taken = out >= 0
    far = np.abs(x[:, :3] - x[:, 3:]).max(axis=1)
    assert np.all(taken[far >= 2.0 ** (56 - k) * (1 + 2.0 ** -20)]) and not np.any(taken[far < 2.0 ** (56 - k) * (1 - 2.0 ** -20)])
    err = np.abs(out[taken].astype(np.longdouble) / want[taken] - 1)
    t = max(kappa, 0) / scale * r[taken]
    assert np.all(err <= 1.2e-16 + np.sqrt(3.0) * 2.0 ** -56 * (1 + t) + t * 1.45 * 2.0 ** -58)
    assert taken[:2].all()
