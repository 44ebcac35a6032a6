"""Device functions of the kernels' sources, compiled for the host: a test names functions of a
.cuh file, their text is taken from the file and built by g++ with the packed and approximate
operations stated in plain C++ (correctly rounded where the GPU's are approximate), one lane to a
warp. So what a function does with a number, and with one that is none, can be looked at on the CPU."""
import ctypes
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_20787_gb300", "csrc")

PRELUDE = r"""
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
using std::max; using std::min;
typedef unsigned long long u64;
static u64 pk(float a, float b) { u64 r; float v[2] = {a, b}; memcpy(&r, v, 8); return r; }
static void upk(u64 r, float& a, float& b) { float v[2]; memcpy(v, &r, 8); a = v[0]; b = v[1]; }
#define PACKED(name, expr) static u64 name(u64 x, u64 y) { float a, b, c, d; upk(x, a, b); upk(y, c, d); \
  float v[2]; { float p = a, q = c; v[0] = expr; } { float p = b, q = d; v[1] = expr; } return pk(v[0], v[1]); }
PACKED(add2, p + q) PACKED(sub2, p - q) PACKED(mul2, p * q)
static u64 fma2(u64 x, u64 y, u64 z) {
  float a, b, c, d, e, f; upk(x, a, b); upk(y, c, d); upk(z, e, f); return pk(fmaf(a, c, e), fmaf(b, d, f)); }
static float ftz(float x) { return fabsf(x) < 1.17549435e-38f ? copysignf(0.0f, x) : x; }
static float rsq(float x) { x = ftz(x); return ftz((float)(1.0 / sqrt((double)x))); }
static float rcp_approx(float x) { x = ftz(x); return ftz((float)(1.0 / (double)x)); }
static int __float_as_int(float x) { int r; memcpy(&r, &x, 4); return std::isnan(x) ? 0x7fffffff : r; }
static float __uint_as_float(unsigned x) { float r; memcpy(&r, &x, 4); return r; }
static int __reduce_max_sync(unsigned, int v) { return v; }
static bool __any_sync(unsigned, bool v) { return v; }
"""


def function(file, name):
    """The text of a device function (with its template line), host-compilable."""
    src = open(os.path.join(CSRC, file)).read()
    m = re.search(r"(?:template <[^\n]*>\n)?[^\n]*__device__[^\n]*\b%s\(" % name, src)
    at = src.index("{", m.end())
    depth, end = 0, at
    while True:
        depth += {"{": 1, "}": -1}.get(src[end], 0)
        end += 1
        if depth == 0:
            break
    text = re.sub(r"__(?:host|device|forceinline|noinline)__ ", "", src[m.start():end])
    text = re.sub(r"asm\(\"sqrt\.approx\.ftz\.f32 %0, %1;\" : \"=f\"\((\w+)\) : \"f\"\((.*?)\)\);", r"\1 = sqrtf(\2);",
                  text)
    return text if text.lstrip().startswith(("static", "template", "constexpr")) else "static " + text


def parameters(file, name):
    """Names of a function's parameters."""
    src = open(os.path.join(CSRC, file)).read()
    m = re.search(r"__device__[^\n]*\b%s\((.*?)\)\s*\{" % name, src, re.S)
    return [p.split()[-1].lstrip("&*") for p in m.group(1).split(",")]


def constants(file, *names):
    src = open(os.path.join(CSRC, file)).read()
    return "\n".join(re.search(r"^constexpr [^\n]*\b%s = [^\n]*;" % n, src, re.M).group(0).split("//")[0] for n in names)


def compile_host(directory, *parts):
    path = os.path.join(str(directory), "device_source")
    with open(path + ".cpp", "w") as f:
        f.write(PRELUDE + "\n".join(parts))
    subprocess.run(["g++", "-O1", "-ffp-contract=off", "-std=c++17", "-w", "-shared", "-fPIC", "-o", path + ".so",
                    path + ".cpp"], check=True)
    return ctypes.CDLL(path + ".so")
