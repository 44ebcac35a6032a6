"""The FP64 form's closed window (window64 in pair_fp64.cuh, its text built for the CPU) against the
image sums in extended precision: a pair's force is on average no further from them than the walk of
the images in FP64 is, for every window that takes the closed form and wherever the pair lies."""
import ctypes
import re

import numpy as np
import pytest

import device_source as ds

WORDS = r"""
static long long __double_as_longlong(double x) { long long r; memcpy(&r, &x, 8); return r; }
static double __longlong_as_double(long long x) { double r; memcpy(&r, &x, 8); return r; }
static int __double2hiint(double x) { return (int)(__double_as_longlong(x) >> 32); }
static int __double2loint(double x) { return (int)__double_as_longlong(x); }
static double __hiloint2double(int h, int l) { return __longlong_as_double(((long long)h << 32) | (unsigned)l); }
static unsigned __float_as_uint(float x) { unsigned r; memcpy(&r, &x, 4); return r; }
static double seed(double x) { return __hiloint2double(__double2hiint(x), 0); }  // 20 bits
using std::fabs; using std::sqrt;
"""
RUN = r"""
extern "C" int first() { return kLineMin64; }
template <class T> static void walk(T d2, T dz, T h, int n_cut, T& R, T& Z) {
  R = Z = 0;
  auto image = [&](T o) {
    const T r2 = fma(o, o, d2), r = sqrt(r2), ri = 1 / r, u = r / h, h3 = h * h * h;
    T f = ri * ri * ri;
    if (u < T(0.5)) f = (T(32) / 3 + u * u * (32 * u - T(192) / 5)) / h3;
    else if (u < 1) f = (T(64) / 3 - 48 * u + T(192) / 5 * u * u - T(32) / 3 * u * u * u - 1 / (15 * u * u * u)) / h3;
    R += f;
    Z = fma(o, f, Z);
  };
  image(dz);
  for (int k = 1; k < n_cut; ++k) { image(dz + k); image(dz - k); }
  if (dz != 0) image(dz - std::copysign((T)n_cut, dz));
}
extern "C" void run(int n, const double* d2, const double* dz, double h, int n_cut, double* out, double* walked, double* err) {
  for (int i = 0; i < n; ++i) {
    double r, z, a, b;
    long double R, Z;
    window64<kPair64Line>(d2[i], dz[i], h, n_cut, r, z);
    walk<double>(d2[i], dz[i], h, n_cut, a, b);
    walk<long double>(d2[i], dz[i], h, n_cut, R, Z);
    const long double size = d2[i] * R * R + Z * Z;
    out[i] = sqrtl((d2[i] * (r - R) * (r - R) + (z - Z) * (z - Z)) / size);
    walked[i] = sqrtl((d2[i] * (a - R) * (a - R) + (b - Z) * (b - Z)) / size);
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    src = open(ds.CSRC + "/pair_fp64.cuh").read()
    body = src[src.index("// ---- words"):src.index("// dz wrapped to")]
    body = re.sub(r"__(?:host|device|forceinline|noinline)__ ", "", body)
    body = re.sub(r'asm\("rsqrt\.approx\.ftz\.f64 [^)]*\) : "d"\((\w+)\)\);', r"y = seed(1.0 / sqrt(\1));", body)
    body = re.sub(r'asm\("rcp\.approx\.ftz\.f64 [^)]*\) : "d"\((\w+)\)\);', r"y = seed(1.0 / \1);", body)
    lib = ds.compile_host(tmp_path_factory.mktemp("fp64"), WORDS, body, RUN)
    lib.run.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_double, ctypes.c_int] + [ctypes.c_void_p] * 3
    return lib


@pytest.mark.parametrize("h", [1e-4, 0.3, 3.0])
@pytest.mark.parametrize("lo,hi", [(0.1, 1.0), (1.0, 4.0), (4.0, 15.9)])
@pytest.mark.parametrize("n_cut", [0, 1, 2, 8, 48, 80])  # beyond the first that takes the closed form
def test_no_further_off_than_the_walk(lib, n_cut, lo, hi, h):
    n_cut += lib.first()
    rng = np.random.default_rng(n_cut)
    n = 4000
    d2 = (10 ** rng.uniform(np.log10(lo), np.log10(hi), n)) ** 2
    dz = rng.uniform(-0.5, 0.5, n)
    out, walked = np.zeros(n), np.zeros(n)
    lib.run(n, d2.ctypes.data, dz.ctypes.data, h, n_cut, out.ctypes.data, walked.ctypes.data, None)
    assert np.sqrt((out ** 2).mean()) <= np.sqrt((walked ** 2).mean())
    assert out.max() <= 32 * 2.0 ** -52
