"""Which loads the two-word fixed-point sums take (fix_bound, fix_resolves in
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
extern "C" int resolves(double B, double M, double m, double D, int n, double most) { return fix_resolves(B, M, m, D, n, most); }
extern "C" double limit(int fp32) { return fp32 ? kMaxSpreadF : kMaxSpread; }
extern "C" int bits() { return kLoBits; }
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    lib = ds.compile_host(tmp_path_factory.mktemp("fix"), ds.constants("pair_sym.cuh", "kLoBits", "kMaxSpread"),
                          ds.function("pair_sym.cuh", "fix_bound"), ds.function("pair_sym.cuh", "fix_resolves"), WRAP)
    d = ctypes.c_double
    lib.bound.argtypes, lib.bound.restype, lib.limit.restype = [d, d, ctypes.c_int], d, d
    lib.resolves.argtypes = [d, d, d, d, ctypes.c_int, d]
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
    spread = B / (m.sum() - m.max()) * (D * np.hypot(D, n_cut) / (2 * n_cut) if n_cut else D * D)
    got = two_word(t, np.longdouble(2) ** np.floor(57 - np.log2(B)), rule.bits())
    err = np.linalg.norm(got - exact, axis=1) / np.linalg.norm(exact, axis=1)
    # one unit is at most 2^-96 B (a power of two below 2^57 / B); a particle's sum rounds once per
    # term, half a unit each, in three components
    unit = 2.0 ** -96 * spread * 2 * np.sqrt(3 * t.shape[1])
    for fp32 in (0, 1):
        most = rule.limit(fp32)
        taken = rule.resolves(B, m.sum(), m.max(), D, n_cut, most)
        assert not taken or spread <= most
        if taken:  # FP64's rounding of a sum is 1.1e-16, FP32's 6e-8
            assert np.median(err) <= unit and err[0] <= 30 * unit and unit <= (1e-12 if fp32 else 1e-17)
        # what does not depend on the units: a load with an ordinary softening is accepted
        if soft >= (1e-7 if fp32 else 1e-3) and not heavy and (n_cut == 0 or R == 1.0):
            assert taken


def test_the_rule_has_no_units(rule):
    def largest(n_cut, M, length):  # the largest L / h that is taken
        lo, hi = 1.0, 1e12
        for _ in range(80):
            q = np.sqrt(lo * hi)
            ok = rule.resolves(rule.bound(M, q / length, int(n_cut > 0)), M, 0.25 * M, 3.0 * length, n_cut, rule.limit(0))
            lo, hi = (q, hi) if ok else (lo, q)
        return lo
    for n_cut in (0, 16):
        a = largest(n_cut, 1.0, 1.0)
        assert a > 1e3 and abs(largest(n_cut, 1e-9, 1.0) - a) <= 1e-9 * a
    assert abs(largest(0, 1.0, 1e6) - largest(0, 1.0, 1.0)) <= 1e-9 * a
