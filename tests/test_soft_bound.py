"""The softened images beyond the near ones (far_soft2 in pair2.cuh, up to the bound of soft_bound2),
from their source on the CPU. Over the infinite window no image number ends them but the bound, so no
position, whatever its bits, may take the walk beyond rn(h), the last image that a support of h can
reach from |dz| <= 1/2; and every softened image has to be walked."""
import ctypes
import itertools
import struct

import numpy as np
import pytest

import device_source as ds

NAMES = ["dup", "rsq2", "rcp2", "max2", "neg2", "inv_r3", "flag_nonzero2"]
WRAP = r"""
extern "C" int far(float h, float d, float a, float g, float e, float b, int m, int n_cut, float* out) {
  const u64 HH = pk(h, g), H2 = mul2(HH, HH), DR2 = pk(d, e), ADZ = pk(a, b);
  const Soft2 s = soft2(HH);
  const int kw = soft_bound2(H2, DR2, ADZ);
  u64 SR = 0, SZ = 0;
  images = 0;
  try { if (kw > m) { CALL } } catch (int) {}
  upk(SR, out[0], out[1]);
  upk(SZ, out[2], out[3]);
  return images / 2;  // both sides of each
}
"""
LIMIT = 100000


@pytest.fixture(scope="module")
def far(tmp_path_factory):
    neg = "constexpr u64 kSign2 = 0x8000000080000000ull;"
    count = "static int images;"
    inv = ds.function("pair2.cuh", "inv_r3").replace("{", "{ if (++images > %d) throw 1;" % (2 * LIMIT), 1)
    src = open(ds.CSRC + "/pair2.cuh").read()
    soft = src[src.index("struct Soft2 {"):src.index("};", src.index("struct Soft2 {")) + 2]
    reach = [ds.function("pair2.cuh", "soft_reach2")] if "soft_reach2" in src else []
    args = ", ".join(ds.parameters("pair2.cuh", "far_soft2"))
    call = "far_soft2(%s);" % args
    if ds.function("pair2.cuh", "far_soft2").startswith("template"):
        call = "if (n_cut) far_soft2<false>(%s); else far_soft2<true>(%s);" % (args, args)
    lib = ds.compile_host(tmp_path_factory.mktemp("far"), neg, count,
                          ds.constants("pair_fp32.cuh", "kTwo23", "kTwo23Bits"),
                          *[inv if n == "inv_r3" else ds.function("pair2.cuh", n) for n in NAMES], soft,
                          ds.function("pair2.cuh", "soft2"), ds.function("pair_fp32.cuh", "spline_outer_value"),
                          ds.function("pair_fp32.cuh", "spline_value_r2"), ds.function("pair2.cuh", "spline2"),
                          ds.function("pair2.cuh", "soft_bound2"), *reach, ds.function("pair2.cuh", "far_soft2"),
                          WRAP.replace("CALL", call))
    lib.far.argtypes = [ctypes.c_float] * 6 + [ctypes.c_int] * 2 + [ctypes.c_void_p]

    def run(*args):
        out = np.zeros(4, np.float32)
        return lib.far(*args, out.ctypes.data), out
    return run


def exact(h, d2, adz, m, top):
    """Spline minus Newtonian of the images m < |k| <= top, and the size of the terms."""
    h, d2, adz = (np.float64(np.float32(v)) for v in (h, d2, adz))
    sr = sz = size = 0.0
    for k in range(m + 1, top + 1):
        for o in (adz - k, adz + k):
            r = np.sqrt(o * o + d2)
            u = r / h
            if u < 0.5:
                f = (32 / 3 + u * u * (32 * u - 38.4)) / h ** 3
            elif u < 1:
                f = (64 / 3 - 48 * u + 38.4 * u * u - 32 / 3 * u ** 3 - 1 / (15 * u ** 3)) / h ** 3
            else:
                continue
            f -= r ** -3
            sr, sz, size = sr + f, sz + o * f, size + r ** -3 * max(1.0, abs(o))
    return sr, sz, size


NAN, INF = float("nan"), float("inf")
NEG_NAN = struct.unpack("f", struct.pack("I", 0xffffffff))[0]


@pytest.mark.parametrize("adz,d2", list(itertools.product([0.0, 0.5, NAN, NEG_NAN, INF, 1e30], [0.0, 0.04, NAN, INF])))
@pytest.mark.parametrize("h", [0.01, 0.5, 3.0, 17.3, 1000.0])
def test_no_position_takes_the_walk_beyond_the_support(far, adz, d2, h):
    # beside a pair with a softened tail, which keeps its sums
    for m, args in ((3, (6.2, 1.5, 0.3, h, d2, adz)), (3, (h, d2, adz, 6.2, 1.5, 0.3)), (0, (h, d2, adz, h, d2, adz))):
        images, out = far(*args, m, 0)
        assert images <= int(max(np.rint(h), 6))
        if m:
            q = 0 if args[0] == 6.2 else 1
            sr, sz, size = exact(6.2, 1.5, 0.3, m, 6)
            # 4 e-7: some six roundings of each image's spline and of the sums
            assert abs(out[q] - sr) <= 4e-7 * size and abs(out[2 + q] - sz) <= 4e-7 * size


def test_every_softened_image_is_walked(far):
    rng = np.random.default_rng(5)
    for _ in range(500):
        h, adz = np.float32(10 ** rng.uniform(-1, 1.7)), np.float32(rng.choice([0.0, 0.5, rng.uniform(0, 0.5)]))
        d2 = np.float32((h * rng.uniform(0, 1.2)) ** 2)
        for n_cut in (0, 12):
            top = 100 if n_cut == 0 else n_cut - 1
            images, out = far(h, d2, adz, 0.1, 1.0, 0.2, 3, n_cut)
            if n_cut and images > n_cut - 4:
                continue  # the window's edge image is among them
            sr, sz, size = exact(h, d2, adz, 3, top)
            assert abs(out[0] - sr) <= 4e-7 * size and abs(out[2] - sz) <= 4e-7 * size, (h, adz, d2, n_cut)
