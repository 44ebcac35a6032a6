"""Which loads the two-word fixed-point sums take (fix_bound, fix_spread and their limit in
pair_sym.cuh, built from the source for the CPU), and that the sums they accept lose nothing: the
kernels' terms (one FP32 sum per particle and block of 128) are rounded to the accumulator's unit and
added up, for total masses from 1e-12 to 1e12, radii from 1 to 1e8 of the unit of length, and a
particle 1e9 times as heavy as the others."""
import ctypes

import numpy as np
import pytest

import device_source as ds

WRAP = """
extern "C" double bound(double M, double q, int images) { return fix_bound(M, q, images != 0); }
extern "C" double spread(double B, double M, double m, double D, int n) { return fix_spread(B, M, m, D, n); }
extern "C" double limit() { return kMaxSpread; }
extern "C" int bits() { return kLoBits; }
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    lib = ds.compile_host(tmp_path_factory.mktemp("fix"), ds.constants("pair_sym.cuh", "kLoBits", "kMaxSpread"),
                          ds.function("pair_sym.cuh", "fix_bound"), ds.function("pair_sym.cuh", "fix_spread"), WRAP)
    d = ctypes.c_double
    for f, a in ((lib.bound, [d, d, ctypes.c_int]), (lib.spread, [d, d, d, d, ctypes.c_int]), (lib.limit, [])):
        f.argtypes, f.restype = a, d
    return lib


def terms(pos, m, h, n_cut):
    """[i][block][3]: the sums over each 128 j, in FP32."""
    d = pos[:, None] - pos[None]
    hh = h[:, None] + h[None]
    def f(o, r2):  # of the spline its size is what counts
        return np.where(r2 < hh * hh, 1.0 / hh ** 3, 1.0 / np.maximum(r2, 1e-150) ** 1.5)
    if n_cut == 0:
        v = d * f(d[..., 2], (d * d).sum(-1))[..., None]
    else:
        R2 = (d[..., :2] ** 2).sum(-1)
        dz = d[..., 2] - np.rint(d[..., 2])
        o = [dz + k for k in range(-n_cut + 1, n_cut)]
        F = [f(q, R2 + q * q) for q in o]
        v = np.stack([d[..., 0] * sum(F), d[..., 1] * sum(F), sum(q * g for q, g in zip(o, F))], -1)
    v = v * m[None, :, None]
    return np.stack([v[:, a:a + 128].sum(1) for a in range(0, len(m), 128)], 1).astype(np.float32).astype(np.longdouble)


def two_word(t, scale, bits):
    q = t * scale
    hi = np.rint(q)
    return (hi.sum(1) + np.rint((q - hi) * np.longdouble(2) ** bits).sum(1) / np.longdouble(2) ** bits) / scale


@pytest.mark.parametrize("n_cut", [0, 16])
@pytest.mark.parametrize("M", [1e-12, 1e-6, 1.0, 1e12])
@pytest.mark.parametrize("R", [1.0, 1e4, 1e8])
@pytest.mark.parametrize("soft", [0.05, 1e-3, 1e-7, 1e-9])
@pytest.mark.parametrize("heavy", [False, True])
def test_accepted_sums_lose_nothing(rule, n_cut, M, R, soft, heavy):
    rng = np.random.default_rng(2)
    n = 400
    pos = rng.normal(size=(n, 3)) * R / 3
    if n_cut:
        pos[:, 2] = rng.uniform(0, 1, n)
    m = np.full(n, 1.0 / n)
    if heavy:
        m[1:] *= 1e-9
    m *= M / m.sum()
    h = np.full(n, soft * (R if n_cut == 0 else 1.0))
    B = rule.bound(m.sum(), 1.0 / h.min(), int(n_cut > 0))
    t = terms(pos, m, h, n_cut)
    exact = t.sum(1)
    assert abs(exact).max() <= 16 * B  # 2^57 / B leaves no sum beyond 2^62
    D = 2 * np.sqrt((pos[:, :2 if n_cut else 3] ** 2).sum(1)).max()
    spread = rule.spread(B, m.sum(), m.max(), D, n_cut)
    got = two_word(t, np.longdouble(2) ** np.floor(57 - np.log2(B)), rule.bits())
    err = np.linalg.norm(got - exact, axis=1) / np.linalg.norm(exact, axis=1)
    # one unit is at most 2^-96 B (a power of two below 2^57 / B); a particle's sum rounds once per
    # term, half a unit each, in three components
    unit = 2.0 ** -96 * spread * 2 * np.sqrt(3 * t.shape[1])
    if spread <= rule.limit():  # FP64's rounding of a sum is 1.1e-16
        assert np.median(err) <= unit and err[0] <= 30 * unit and unit <= 1e-17
    # what does not depend on the units: a load with an ordinary softening is accepted
    if soft >= 1e-3 and not heavy and (n_cut == 0 or R == 1.0):
        assert spread <= rule.limit()


def test_spread_has_no_units(rule):
    for n_cut in (0, 16):
        a = rule.spread(rule.bound(1.0, 50.0, int(n_cut > 0)), 1.0, 0.25, 3.0, n_cut)
        b = rule.spread(rule.bound(1e-9, 50.0, int(n_cut > 0)), 1e-9, 0.25e-9, 3.0, n_cut)
        assert abs(a - b) <= 1e-12 * a
    c = rule.spread(rule.bound(1.0, 50.0 / 1e6, 0), 1.0, 0.25, 3.0e6, 0)
    assert abs(c - rule.spread(rule.bound(1.0, 50.0, 0), 1.0, 0.25, 3.0, 0)) <= 1e-12 * c
