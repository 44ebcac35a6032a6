"""The closed form of the image line's far part (pair2.cuh), read from the kernel's
source and evaluated with FP32 numpy arithmetic on the CPU, against the image sums in
FP64: the plain window's for every kind of n_cut it is taken for, the infinite line, and
the modelled tails' near images and continuum base. The bounds are those the source
states (8e-8 of the sum of f, 5e-8 of (x^2 + dR^2)^(-1/2) at the near end, the far ends'
6e-8 at n_cut = 12 and 1e-8 from 16 on) plus 4e-7 of the terms' size for the FP32
arithmetic around the polynomials."""
import os
import re

import numpy as np
import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_20787_gb300", "csrc",
                   "pair2.cuh")
f32 = np.float32
A = 3.5


def polynomial(name):
    """The body of a device polynomial of (Q, D2) as a Python function on FP32 arrays."""
    body = re.search(r"u64 %s\(u64 Q, u64 D2\) \{(.*?)\n\}" % name, open(SRC).read(), re.S).group(1)
    body = re.sub(r"(\d)f\b", r"\1", body).replace("u64 ", "").replace(";", "")
    lines = [ln.strip() for ln in re.sub(r",\n\s+", ", ", body).strip().splitlines()]

    def run(q, d2):
        env = {"Q": q, "D2": d2, "dup": lambda c: f32(c), "fma2": lambda a, b, c: (a * b + c).astype(f32)}
        for ln in lines:
            if ln.startswith("return"):
                return env["r"]
            exec(ln, {}, env) if "r" in ln else None
    return run


def samples():
    rng = np.random.default_rng(3)
    n = 20000
    R = np.concatenate([[0.0, 1e-4], 10 ** rng.uniform(-2, 3, n), rng.uniform(0, 8, n)])
    dz = rng.uniform(0, 0.5, R.size)
    dz[:4] = [0.0, 0.5, 0.0, 0.5]
    return R.astype(f32), dz.astype(f32)


def side_sums(x, R, top=6000):
    """Images x + 1/2 + j, j >= 0, of f and z f in FP64 (a long sum and two Euler-Maclaurin terms)."""
    sr, sz = np.zeros_like(R), np.zeros_like(R)
    near = 40
    for j in range(near):
        o = x + 0.5 + j
        f = (o * o + R * R) ** -1.5
        sr += f
        sz += o * f
    x = x + near
    i = 1 / np.sqrt(x * x + R * R)
    s, e = x * i, i * i
    return (sr + e / (1 + s) - s * e * e / 8 + 7 / 384 * s * e ** 3 * (7 * s * s - 3),
            sz + i + i ** 3 * (1 - 3 * s * s) / 24 + 7 / 1920 * i ** 5 * (35 * s ** 4 - 30 * s * s + 3))


def closed(kind, R, dz, N=None):
    T, Z = polynomial(kind + "_poly_r"), polynomial(kind + "_poly_z")
    r2 = (R * R).astype(f32)
    il = (1 / np.sqrt(r2 + f32(A * A))).astype(f32)
    s, e = (il * f32(A)).astype(f32), (il * il).astype(f32)
    q, d2, g = (s * s).astype(f32), (dz * dz).astype(f32), (s * e).astype(f32)
    if N is None:
        I, z = 2 * e / (s + f32(1)), f32(0)
    else:
        ih = (1 / np.sqrt(r2 + f32(N * N))).astype(f32)
        sn, en = (ih * f32(N)).astype(f32), (ih * ih).astype(f32)
        d = dz - f32(0.5)
        dd, gn = d * d, sn * en
        I = f32(2 * (N * N - A * A)) * e * en / (s + sn) + gn * en * (f32(0.25) - f32(3) * dd)
        z = d * gn * (f32(2) + en * (f32(9) - f32(15) * sn * sn) * (f32(1 / 12) - dd / f32(3)))
    return (g * e * T(q, d2) + I).astype(f32), (dz * g * Z(q, d2) + z).astype(f32)


def check(kind, N, ref_r, ref_z, R, dz):
    sr, sz = closed(kind, R, dz, N)
    far = 0.0 if N is None else 1.1e-8 * (16.0 / N) ** 6
    R, dz = R.astype(float), dz.astype(float)
    i = 1 / np.sqrt(R * R + A * A)
    assert np.all(np.abs(sr - ref_r) <= (8e-8 + 4e-7) * np.abs(ref_r) + far + 2e-7 * i ** 3)
    assert np.all(np.abs(sz - ref_z) <= (5e-8 + 2e-7) * i + far)


@pytest.mark.parametrize("n_cut", [12, 13, 16, 24, 64, 333, 4096])
def test_plain_window(n_cut):
    R, dz = samples()
    r, z = R.astype(float), dz.astype(float)
    ua, za = side_sums(A + z, r)
    ub, zb = side_sums(A - z, r)
    # the closed form holds the edge image at every dz (the kernel takes it off at dz = 0)
    va, wa = side_sums(n_cut - 0.5 + z, r)
    vb, wb = side_sums(n_cut + 0.5 - z, r)
    check("line", n_cut, ua + ub - va - vb, za - zb - wa + wb, R, dz)


def test_infinite_line_and_base():
    R, dz = samples()
    r, z = R.astype(float), dz.astype(float)
    ua, za = side_sums(A + z, r)
    ub, zb = side_sums(A - z, r)
    check("line", None, ua + ub, za - zb, R, dz)
    # the modelled tails' line: image 4 on each side and the base beyond it
    out = []
    for x, o in ((4.5 + z, 4.0 + z), (4.5 - z, 4.0 - z)):
        i = 1 / np.sqrt(x * x + r * r)
        s, e = x * i, i * i
        f = (o * o + r * r) ** -1.5
        out.append((e / (1 + s) - s * e * e / 8 + f, i + i ** 3 * (1 - 3 * s * s) / 24 + o * f))
    check("base", None, out[0][0] + out[1][0], out[0][1] - out[1][1], R, dz)
