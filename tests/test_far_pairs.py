"""Pairs very far apart: the closed far part of the image line (line_far2 and window_walk2 of
pair2.cuh, built from their source for the CPU) against the image sums in FP64, from ordinary
separations to the largest of packed positions (2.9e38 for dR^2; the infinite window's have no cap).
The images' sum falls as 1 / dR^3 and is a normal FP32 number up to dR of some 1e12; beyond it has to end
at zero, as the images one by one do."""
import ctypes

import numpy as np
import pytest

import device_source as ds

WRAP = r"""
extern "C" void run(int kind, float d2, float adz, int n_cut, float* out) {
  const u64 DR2 = dup(d2), ADZ = dup(adz);
  u64 SR = 0, SZ = 0;
  if (kind == 0) { line_far2<false, false, true>(DR2, ADZ, (float)n_cut, SR, SZ); }
  if (kind == 4) { line_far2<false, false>(DR2, ADZ, (float)n_cut, SR, SZ); }
  if (kind == 1) { line_far2<true, false>(DR2, ADZ, 0.0f, SR, SZ); }
  if (kind == 2) { line_far2<false, true>(DR2, ADZ, (float)n_cut, SR, SZ); }
  if (kind == 3) window_walk2<true>(DR2, dup(0.0f), fma2(ADZ, ADZ, DR2), ADZ, false, 8, n_cut, (float)n_cut, SR, SZ);
  if (kind == 5) window_walk2<false>(DR2, dup(0.0f), fma2(ADZ, ADZ, DR2), ADZ, false, 8, n_cut, (float)n_cut, SR, SZ);
  float x;
  upk(SR, out[0], x);
  upk(SZ, out[1], x);
}
"""


@pytest.fixture(scope="module")
def sums(tmp_path_factory):
    src = open(ds.CSRC + "/pair2.cuh").read()
    structs = ["constexpr u64 kSign2 = 0x8000000080000000ull;"]
    for s in ("Soft2", "FarEnd2", "LineSide2"):
        a = src.index("struct %s {" % s)
        structs.append(src[a:src.index("};", a) + 2])
    f2 = ["dup", "rsq2", "rcp2", "max2", "neg2", "inv_r3", "flag_nonzero2", "any_less2", "newton2", "newton_k2", "soft2"]
    lib = ds.compile_host(
        tmp_path_factory.mktemp("far"), *structs, ds.constants("pair_fp32.cuh", "kTwo23", "kTwo23Bits"),
        ds.constants("pair2.cuh", "kPolyA"),
        *[ds.constants("pair2.cuh", k) for k in ("kFarFloor", "kFarUp") if k in src], *[ds.function("pair2.cuh", f) for f in f2],
        ds.function("pair_fp32.cuh", "spline_outer_value"), ds.function("pair_fp32.cuh", "spline_value_r2"),
        *[ds.function("pair2.cuh", f) for f in ("spline2", "soft_bound2", "spline_one2", "spline_centre2", "near_soft_walk2",
                                                "near_newton2", "line_poly_r", "line_poly_z", "base_poly_r", "base_poly_z",
                                                *(["far_rcp2"] if "far_rcp2" in src else []), "far_end2", "fix_dz0", "line_far2", "line_side2", "window_walk2")], WRAP)
    lib.run.argtypes = [ctypes.c_int, ctypes.c_float, ctypes.c_float, ctypes.c_int, ctypes.c_void_p]

    def run(*args):
        out = np.zeros(2, np.float32)
        lib.run(*args, out.ctypes.data)
        return out
    return run


@pytest.mark.parametrize("n_cut", [12, 64, 4096])
def test_window_of_the_symmetric_kernels(sums, n_cut):
    # without the factor: the same bits up to 1e9, and finite and no larger beyond
    for adz in (0.0, 0.25, 0.5):
        for dR in 10.0 ** np.arange(0.5, 9.1, 0.5):
            d2 = np.float32(dR * dR)
            for wide, kind in ((0, 4), (3, 5)):
                a, b = sums(wide, d2, adz, n_cut), sums(kind, d2, adz, n_cut)
                assert np.array_equal(a, b)
        for d2 in (1e19, 1e22, 1e26, 1e30, 1e37, 2.9e38):
            for kind in (4, 5):
                got = sums(kind, d2, adz, n_cut)
                assert np.all(np.abs(got) <= 2 * n_cut * n_cut * min(1e-28, 1.01 * float(np.float32(d2)) ** -1.5)), (d2, got)


@pytest.mark.parametrize("n_cut", [12, 64, 4096])
@pytest.mark.parametrize("kind", [0, 3])
def test_window(sums, kind, n_cut):
    first = 4 if kind == 0 else 0  # line_far2: the images beyond +-3 alone
    for adz in (0.0, 0.25, 0.5):
        adz = np.float64(np.float32(adz))
        k = np.arange(first, n_cut)
        o = np.concatenate([adz - k, (adz + k)[k > 0]])
        if adz > 0 or kind == 0:  # the edge image, which line_far2 holds at every dz
            o = np.append(o, adz - n_cut)
        for dR in 10.0 ** np.arange(0.5, 11.6, 0.5):
            d2 = np.float32(dR * dR)
            f = (o * o + np.float64(d2)) ** -1.5
            got = sums(kind, d2, adz, n_cut)
            # the z sum of a line is smaller than its terms
            assert abs(got[0] - f.sum()) <= 2e-6 * f.sum(), (dR, adz, got, f.sum())
            assert abs(got[1] - (o * f).sum()) <= 2e-6 * (abs(o) * f).sum() + 1e-6 * f.sum(), (dR, adz)
        for d2 in (1e26, 1e30, 1e37, 2.9e38):
            got = sums(kind, d2, adz, n_cut)
            assert np.all(np.abs(got) <= 2 * n_cut * n_cut * min(1e-36, 1.01 * float(np.float32(d2)) ** -1.5)), (d2, got)


def test_infinite_line(sums):
    for kind, n_cut in ((1, 0), (2, 24)):
        for d2 in 10.0 ** np.arange(1, 38.5):
            d2 = np.float32(d2)
            got = sums(kind, d2, 0.3, n_cut)
            assert np.all(np.isfinite(got))
            if kind == 1:  # at large dR the whole line, 2 / dR^2, less seven images
                ref = 2 / np.float64(d2) - 7 * np.float64(d2) ** -1.5
                assert d2 < 1e6 or d2 > 1e37 or abs(got[0] - ref) <= 1e-5 * ref
    assert np.all(np.isfinite(sums(1, np.inf, 0.3, 0)))
