// FP64 pair kernels (the precision study's reference form): window and softening of
// eq. ForceCylindrical and eq. Force_spline_kernel, every quantity of the force in FP64.
//
// What bounds them: the FP64 pipe, 2 lanes per SM and clock (a warp's FP64 instruction
// holds it for 16 cycles), while loads, shuffles, integer and FP32 instructions are free
// beside it. So the kernels spend other instructions wherever one of FP64 is saved:
//   - each unordered pair once (pair_sym_fp64_kernel), added to both particles;
//   - of the window's 2 n_cut images the 2 x 8 + 1 near ones, and both ends of the rest by
//     the midpoint rule's Euler-Maclaurin series: its first three terms (near ends, two at
//     the far ones) in FP64 and the others, together below 2e-10 of the sum, in FP32 from
//     rounded inputs. A pair's force is then closer to the exact one than the walk's for any
//     window that takes this form (rms error in 2^-52, closed form / walk, at dR = 1 .. 4 and
//     4 .. 16: n_cut = 16 0.74 / 1.22 and 0.80 / 0.95, n_cut = 64 0.73 / 2.4 and 0.72 / 2.2);
//   - 1 / r^3 straight from the hardware's 20-bit 1 / r by a two-term series;
//   - comparisons, signs, conversions and the period's wrap on the integer pipe.
// That leaves about 300 FP64 instructions per pair for any n_cut.
#pragma once
#include <cstdint>

#include "pair_sym.cuh"

namespace steps {

// ---- words ------------------------------------------------------------------------
// Order of two doubles >= 0 (a NaN is larger than any number).
__device__ __forceinline__ bool less_pos(double a, double b) {
  return __double_as_longlong(a) < __double_as_longlong(b);
}
// x >= 0 as a float, truncated; below 2^-126: 0, from 2^128 on (and NaN): infinity.
__device__ __forceinline__ float float_trunc(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  if (hi < 0x38100000u) return 0.0f;
  if (hi >= 0x47f00000u) return __uint_as_float(0x7f800000u);
  return __uint_as_float(((hi - 0x38000000u) << 3) | (lo >> 29));
}
// The same, rounded (half up).
__device__ __forceinline__ float float_rn(double x) {
  return float_trunc(__longlong_as_double(__double_as_longlong(x) + (1LL << 28)));
}
// A float as a double; subnormals become 0.
__device__ __forceinline__ double double_of(float x) {
  const unsigned u = __float_as_uint(x), mag = u & 0x7fffffffu;
  if (mag < 0x00800000u) return 0.0;
  return __hiloint2double((int)((u & 0x80000000u) | ((mag >> 3) + 0x38000000u)), (int)(u << 29));
}

// The hardware's approximations (from the upper word, some 20 bits).
__device__ __forceinline__ double rsqrt_seed(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  return y;
}
// 1 / v for v > 0: y0 (1 + e + e^2), e = 1 - v y0 of some 2^-20.
__device__ __forceinline__ double recip(double v) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(v));
  const double e = fma(-v, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
// 1 / sqrt(v) for v > 0: y0 (1 + e / 2 + 3 e^2 / 8), e = 1 - v y0^2.
__device__ __forceinline__ double inv_sqrt(double v) {
  const double y = rsqrt_seed(v), e = fma(-v, y * y, 1.0);
  return fma(y, e * fma(0.375, e, 0.5), y);
}

// ---- one image -----------------------------------------------------------------------
struct Soft64 {
  double hh2, ih, ih3;
};
constexpr double kTinyR2 = 1e-150;  // floor of r^2: keeps the seed and its cube finite
constexpr double kHugeR2 = 1e300;   // its ceiling: keeps the seed's square normal and the series finite

// F / r at r^2 = r2: y0^3 (1 + 3 e / 2 + 15 e^2 / 8) with e = 1 - r^2 y0^2 for 1 / r^3, and
// the spline where soft and r < h.
__device__ __forceinline__ double image64(double r2, bool soft, const Soft64& h) {
  const double y = rsqrt_seed(r2), w = y * y, e = fma(-r2, w, 1.0), y3 = w * y;
  double f = fma(y3, e * fma(1.875, e, 1.5), y3);
  if (soft && less_pos(r2, h.hh2)) {
    const double u = r2 * fma(y, e * fma(0.375, e, 0.5), y) * h.ih;
    if (less_pos(u, 0.5))
      f = fma(u * u, fma(32.0, u, -38.4), 32.0 / 3.0) * h.ih3;
    else
      f = fma(f, -1.0 / 15.0, fma(u, fma(u, fma(u, -32.0 / 3.0, 38.4), -48.0), 64.0 / 3.0) * h.ih3);
  }
  return f;
}

// ---- the ends of the image line ------------------------------------------------------
// With x half-way between two images, r^2 = x^2 + dR^2, i = 1 / r, s = x i, e = i^2,
// q = s^2: the sums of f = 1 / r^3 and z f over the images beyond x are their integrals
// plus s e^(p+1) C_p(q) and i e^p D_p(q), p = 1, 2, ..., the polynomials from the
// derivatives of f and z f and the midpoint rule's coefficients 1/24, -7/5760, 31/967680, ...
// line_rest: the terms from p = 4 on over s e^5 and i e^4, in t = 1 - q (in which
// they cancel least): p = 4 and 5 exact, the rest fitted over x >= 7 (the ends lie at 8 and beyond).
__device__ __forceinline__ void line_rest(float t, float e, float& R, float& Z) {
  const float r0 = fmaf(t, fmaf(t, fmaf(t, -1.66268921f, 2.66030273f), -1.22783203f), 0.148828125f);
  const float r1 = fmaf(t, fmaf(t, fmaf(t, fmaf(t, -13.6419233f, 28.7198385f), -20.2728271f), 5.40608724f), -0.415852865f);
  const float r2 = fmaf(t, fmaf(t, fmaf(t, fmaf(t, fmaf(t, -164.554708f, 426.652138f), -406.970009f), 172.059576f),
                                -30.4928176f), 1.63194019f);
  const float r3 = fmaf(t, fmaf(t, fmaf(t, fmaf(t, fmaf(t, 3621.42496f, -6304.90564f), 4209.46417f), -1297.91088f),
                                173.135063f), -7.09924357f);
  R = fmaf(e, fmaf(e, fmaf(e, r3, r2), r1), r0);
  const float z0 = fmaf(t, fmaf(t, fmaf(t, fmaf(t, 1.66268921f, -3.54707031f), 2.45566406f), -0.5953125f), 0.0330729167f);
  const float z1 = fmaf(t, fmaf(t, fmaf(t, fmaf(t, fmaf(t, 13.6419233f, -35.8997981f), 33.7880452f), -13.5152181f),
                                2.07926432f), -0.0756096117f);
  const float z2 = fmaf(t, fmaf(t, fmaf(t, fmaf(t, fmaf(t, fmaf(t, 159.011736f, -501.49549f), 602.922408f), -341.568994f),
                                        91.0711901f), -9.76574712f), 0.251302702f);
  const float z3 = fmaf(t, fmaf(t, fmaf(t, fmaf(t, fmaf(t, fmaf(t, -3747.2272f, 8004.32516f), -6824.68262f), 2858.17171f),
                                        -580.343949f), 48.1405493f), -0.959517899f);
  Z = fmaf(e, fmaf(e, fmaf(e, z3, z2), z1), z0);
}

// An end at x: i, s, e, and the images beyond it without the integral of f: FP64 terms R
// and Z (with z f's integral i), FP32 terms fr and fz. NEAR: p <= 3 in FP64, else p <= 2 (for
// x >= 15, where the third is below 2e-10 of the sum).
struct End64 {
  double s, e, R, Z;
  float fr, fz;
};
template <bool NEAR>
__device__ __forceinline__ End64 line_end64(double x, double dR2, float R2f) {
  End64 E;
  const double i = inv_sqrt(fma(x, x, dR2));
  E.s = x * i;
  E.e = i * i;
  const double q = E.s * E.s, e = E.e;
  // rounded, and each from FP64: the terms are up to tenth powers of their inputs, and inputs cut
  // off at 23 bits left 0.9 of 2^-52 of the sum
  const float fi = float_rn(i), fe = float_rn(e), fs = float_rn(E.s), ft = R2f * fe, fe2 = fe * fe;
  float gr, gz;
  line_rest(ft, fe, gr, gz);
  double c = fma(q, 49.0 / 384.0, -7.0 / 128.0);
  double d = fma(q, fma(q, 49.0 / 384.0, -7.0 / 64.0), 7.0 / 640.0);
  if (NEAR) {
    c = fma(e, fma(q, fma(q, -341.0 / 1024.0, 155.0 / 512.0), -155.0 / 3072.0), c);
    d = fma(e, fma(q, fma(q, fma(q, -341.0 / 1024.0, 465.0 / 1024.0), -155.0 / 1024.0), 155.0 / 21504.0), d);
    E.fr = fs * fe * (fe2 * fe2) * gr;
    E.fz = fi * (fe2 * fe2) * gz;
  } else {
    const float c3 = fmaf(ft, fmaf(ft, -0.333007812f, 0.36328125f), -0.0807291667f);
    const float d3 = fmaf(ft, fmaf(ft, fmaf(ft, 0.333007812f, -0.544921875f), 0.2421875f), -0.0230654762f);
    E.fr = fs * (fe2 * fe2) * fmaf(fe, gr, c3);
    E.fz = fi * fe * fe2 * fmaf(fe, gz, d3);
  }
  E.R = E.s * e * e * fma(e, c, -0.125);
  E.Z = fma(i * e, fma(e, d, fma(q, -0.125, 1.0 / 24.0)), i);
  return E;
}

// ---- the window ------------------------------------------------------------------------
// Near images of the closed form, and the n_cut it is taken from. Eight is the fewest for
// which a pair's error is no larger than the walk's from dR = 4 on as well (seven: 0.98 against 0.95 of 2^-52,
// n_cut = 16). The walk of a window of 15 images takes as many FP64 instructions as the closed form; from
// n_cut = 16 on the far ends lie at 15 or beyond. Beyond dR = 16 the window is walked: there the sums'
// integrals, of order 1 / dR^2 and 1 / dR, would cancel for a short window.
constexpr int kNear64 = 8;
constexpr int kLineMin64 = 16;
constexpr double kLineMaxR2 = 256.0;
__host__ __device__ __forceinline__ bool line_form64(int n_cut) { return n_cut >= kLineMin64; }

enum Pair64 { kPair64Walk, kPair64Line, kPair64R3 };

// SR = sum F / r, SZ = sum o F / r over the window |dz + k| < n_cut, at the separation dR2, dz
// (|dz| <= 1/2), softening sum hh. A pair's bits do not depend on its warp. kPair64R3: the
// one image of the R^3 force.
template <int KIND>
__device__ __forceinline__ void window64(double dR2, double dz, double hh, int n_cut, double& SR, double& SZ) {
  const double adz = fabs(dz);
  if (less_pos(kHugeR2, dR2)) dR2 = kHugeR2;  // a NaN stays one in dx or dy
  Soft64 h;
  h.hh2 = hh * hh;
  h.ih = h.ih3 = 0.0;
  const double c2 = fma(adz, adz, dR2);
  double r2c = less_pos(c2, kTinyR2) ? kTinyR2 : c2;
  if (KIND == kPair64R3 && less_pos(kHugeR2, r2c)) r2c = kHugeR2;
  const bool soft = less_pos(c2, h.hh2);
  int m = KIND == kPair64Line ? kNear64 : n_cut - 1;
  float R2f = 0.0f;
  if (KIND == kPair64Line) {
    R2f = float_rn(dR2);
    if (!less_pos(dR2, kLineMaxR2)) m = n_cut - 1;
  }
  if (soft) {
    h.ih = recip(hh);
    h.ih3 = h.ih * h.ih * h.ih;
    if (KIND == kPair64Line) {
      // the last k whose image |dz| - k can lie inside the support, or one more
      const float H2f = float_trunc(h.hh2);
      const float kw = float_trunc(adz) + 1.000001f * sqrtf(fmaxf(H2f - R2f, 0.0f) + 4e-7f * H2f) + 1e-5f;
      m = max(m, min((int)fminf(kw, 1e9f), n_cut - 1));
    }
  }
  const double CR = image64(r2c, soft, h);
  SR = CR;
  if (KIND == kPair64R3) {
    SZ = dz * SR;
    return;
  }
  // images +-k: r^2 from (c2 + k^2) -+ 2 k |dz| beyond the first, and the z sum as
  // |dz| sum f + sum k (f+ - f-): one FP64 operation less each
  double SK = 0.0;
  auto images = [&](double k, double rp, double rm) {
    const double fp = image64(rp, soft, h), fm = image64(rm, soft, h);
    SR += fp + fm;
    SK = fma(k, fp - fm, SK);
  };
  if (KIND == kPair64Line || n_cut > 1) {
    const double op = adz + 1.0, om = adz - 1.0;
    images(1.0, fma(op, op, dR2), fma(om, om, dR2));
  }
  int k = 2;
  if (KIND == kPair64Line) {
#pragma unroll
    for (int j = 2; j <= kNear64; ++j) {
      const double b = c2 + (double)(j * j);
      images((double)j, fma(2.0 * j, adz, b), fma(-2.0 * j, adz, b));
    }
    k = kNear64 + 1;
  }
  double fk = KIND == kPair64Line ? kNear64 + 1.0 : 2.0;
#pragma unroll 1
  for (; k <= m; ++k, fk += 1.0) {
    const double op = adz + fk, om = adz - fk;
    images(fk, fma(op, op, dR2), fma(om, om, dR2));
  }
  SZ = fma(adz, SR, SK);
  const bool zero = __double_as_longlong(adz) == 0;  // dz = 0: the window has no edge image
  if (KIND == kPair64Walk || m == n_cut - 1) {
    const double o = adz - (double)n_cut;
    const double f = image64(fma(o, o, dR2), soft, h);
    if (!zero) {
      SR += f;
      SZ = fma(o, f, SZ);
    }
  } else {
    double A = kNear64 + 0.5;
    if (m != kNear64) A = (double)m + 0.5;
    const double kn = zero ? (double)(n_cut - 1) : (double)n_cut;  // the last image below
    const double Xa = ((double)n_cut - 0.5) + adz, Xb = (kn + 0.5) - adz;
    const End64 a = line_end64<true>(A + adz, dR2, R2f), b = line_end64<true>(A - adz, dR2, R2f);
    const End64 fa = line_end64<false>(Xa, dR2, R2f), fb = line_end64<false>(Xb, dR2, R2f);
    // the integrals of f, (X^2 - x^2) e_x e_X / (s_x + s_X), over one denominator
    const double ca = (double)(n_cut - 1 - m), cb = zero ? ca : ca + 1.0;
    const double na = ca * (a.e * fa.e) * fma(2.0, adz, (double)(n_cut + m));
    const double nb = cb * (b.e * fb.e) * fma(-2.0, adz, kn + (double)(m + 1));
    const double va = a.s + fa.s, vb = b.s + fb.s;
    SR += fma(na, vb, nb * va) * recip(va * vb);
    SR += (a.R + b.R) - (fa.R + fb.R);
    SZ += (a.Z - b.Z) - (fa.Z - fb.Z);
    SR += double_of((a.fr + b.fr) - (fa.fr + fb.fr));
    SZ += double_of((a.fz - b.fz) - (fa.fz - fb.fz));
  }
  SZ = __longlong_as_double(__double_as_longlong(SZ) ^ (__double_as_longlong(dz) & (1LL << 63)));
}

// dz wrapped to [-1/2, 1/2], for |dz| <= 1 (dz - rint(dz)).
__device__ __forceinline__ double wrap64(double dz) {
  const long long b = __double_as_longlong(dz), mag = b & 0x7fffffffffffffffLL;
  const long long one = mag > 0x3fe0000000000000LL ? ((b & (1LL << 63)) | 0x3ff0000000000000LL) : 0;
  return dz - __longlong_as_double(one);
}

// ---- rows against every j ------------------------------------------------------------
// Listed particles (idx == nullptr: i = q). CTA (bx, by) takes i-particles [bx * 128, +128)
// against j-tiles [by * tpc, (by + 1) * tpc) of 128 j staged in shared memory, so that a
// short list still fills the GPU; part[by][3][ni] receives the partial sums, which
// chunk_sum_kernel adds in chunk order. The sums are sum_j m_j (dx, dy, dz-part) in units
// of G / L^2, as the FP32 ones.
template <int KIND>
__global__ void __launch_bounds__(128)
pair_fp64_kernel(const double* __restrict__ x, const double* __restrict__ y, const double* __restrict__ z,
                 const double* __restrict__ m, const double* __restrict__ h, int n,
                 const int64_t* __restrict__ idx, int ni, double invL, int n_cut, int tpc,
                 double* __restrict__ part) {
  __shared__ double sx[128], sy[128], sz[128], sm[128], sh[128];
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  const int qq = min(q, ni - 1);
  const int i = idx ? (int)idx[qq] : qq;
  const double xi = x[i] * invL, yi = y[i] * invL, zi = z[i] * invL, hi = h[i] * invL;
  const int NT = (n + 127) / 128;
  const int t0 = blockIdx.y * tpc, t1 = min(NT, t0 + tpc);
  double ax = 0.0, ay = 0.0, az = 0.0;
  for (int t = t0; t < t1; ++t) {
    __syncthreads();
    const int jl = t * 128 + threadIdx.x;
    if (jl < n) {
      sx[threadIdx.x] = x[jl] * invL;
      sy[threadIdx.x] = y[jl] * invL;
      sz[threadIdx.x] = z[jl] * invL;
      sm[threadIdx.x] = m[jl];
      sh[threadIdx.x] = h[jl] * invL;
    }
    __syncthreads();
    const int jn = min(128, n - t * 128);
#pragma unroll 1
    for (int k = 0; k < jn; ++k) {
      if (t * 128 + k == i) continue;
      const double dx = xi - sx[k], dy = yi - sy[k];
      double dz = zi - sz[k];
      if (KIND != kPair64R3) dz = wrap64(dz);
      double SR, SZ;
      if (KIND == kPair64R3)
        window64<KIND>(fma(dx, dx, dy * dy), dz, hi + sh[k], 1, SR, SZ);
      else
        window64<KIND>(fma(dx, dx, dy * dy), dz, hi + sh[k], n_cut, SR, SZ);
      const double ms = sm[k] * SR;
      ax = fma(dx, ms, ax);
      ay = fma(dy, ms, ay);
      az = fma(sm[k], SZ, az);
    }
  }
  if (q < ni) {
    double* dst = part + (long long)blockIdx.y * 3 * ni;
    dst[q] = ax;
    dst[ni + q] = ay;
    dst[2 * (long long)ni + q] = az;
  }
}

// ---- each unordered pair once ------------------------------------------------------------
// Rows and j-slots in blocks of 32, one row per lane; at step s of a pair of blocks lane l
// takes j-slot (l + s) mod 32, so a step is 32 pairs, each i and j once. Block b against
// itself takes the steps 1 .. 16 (16: lower half of the lanes), against a later block 0 .. 31:
// 16 NB^2 steps in all, those of row block b from 16 b (2 NB - b) on. Each warp takes an equal
// contiguous range of steps, so any N splits evenly: at N = 2,048 there are only 2,080 pairs of
// blocks for 608 schedulers. The j side goes round the warp (one 64-bit shuffle per component and step).
//
// Accumulation: as the FP32 kernels, in integers (associative, so the result does not
// depend on the order of the warps), here in two words per sum: hi in units of 1 / scale and
// the remainder in units of 2^-kLoBits / scale (pair_sym.cuh). |lo| stays below 2^39 per term, so
// 2^23 terms fit; scale leaves 2^57 for the bound on |S_i|, so lo resolves 2^-97 of it.
constexpr int kThreads64 = 128;

struct Fix64Acc {
  unsigned long long *hi, *lo;  // [3][n] each
  int n;
  double scale;
  int* err;
};
__device__ __forceinline__ void fix64_add(const Fix64Acc& F, int c, int i, double v) {
  const double q = v * F.scale;
  if (!(fabs(q) < 4.0e18)) {
    atomicOr(F.err, isfinite(v) ? kErrFixRange : kErrNonFinite);
    return;
  }
  const long long a = __double2ll_rn(q), b = __double2ll_rn((q - (double)a) * (double)(1LL << kLoBits));
  const long long o = checked_index((long long)c * F.n + i, 3LL * F.n);
  atomicAdd(F.hi + o, (unsigned long long)a);
  atomicAdd(F.lo + o, (unsigned long long)b);
}
// out[3 n] = the sums as doubles
static __global__ void fix64_sum_kernel(const unsigned long long* __restrict__ hi,
                                        const unsigned long long* __restrict__ lo, long long m, double inv_scale,
                                        double* __restrict__ out) {
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < m; q += (long long)gridDim.x * blockDim.x)
    out[q] = fix_sum(hi[q], lo + q, inv_scale);
}

__host__ __device__ __forceinline__ long long row_step64(int b, int NB) { return 16LL * b * (2LL * NB - b); }
// The row block of step w (row_step64(b) <= w < row_step64(b + 1)).
__device__ __forceinline__ int step_row64(long long w, int NB) {
  int b = NB - (int)ceil(sqrt(fmax((double)NB * NB - (double)w / 16.0, 0.0)));
  b = max(0, min(b, NB - 1));
  while (b > 0 && row_step64(b, NB) > w) --b;
  while (b + 1 < NB && row_step64(b + 1, NB) <= w) ++b;
  return b;
}

template <int KIND>
__global__ void __launch_bounds__(kThreads64)
pair_sym_fp64_kernel(const double* __restrict__ x, const double* __restrict__ y, const double* __restrict__ z,
                     const double* __restrict__ m, const double* __restrict__ h, int n, double invL, int n_cut, int NB,
                     long long W, long long warps, Fix64Acc F) {
  __shared__ double sj[kThreads64 / 32][5][32];
  const int lane = threadIdx.x & 31;
  const long long g = blockIdx.x * (long long)(kThreads64 / 32) + (threadIdx.x >> 5);
  if (g >= warps) return;  // whole warps leave; no block-wide synchronisation follows
  double(*J)[32] = sj[threadIdx.x >> 5];
  long long w = (long long)((double)g / (double)warps * (double)W);
  const long long w1 = g + 1 == warps ? W : (long long)((double)(g + 1) / (double)warps * (double)W);
  while (w < w1) {
    const int b = step_row64(w, NB);
    const long long row0 = row_step64(b, NB), we = min(w1, row_step64(b + 1, NB));
    const int i = b * 32 + lane, ic = min(i, n - 1);
    const double xi = x[ic] * invL, yi = y[ic] * invL, zi = z[ic] * invL, hi = h[ic] * invL;
    const double mi = i < n ? m[ic] : 0.0;  // rows past n repeat the last particle without mass
    double ax = 0.0, ay = 0.0, az = 0.0;
    while (w < we) {
      const long long r = w - row0;
      const bool diag = r < 16;
      const int bj = diag ? b : b + 1 + (int)((r - 16) >> 5);
      const int s0 = diag ? 1 + (int)r : (int)((r - 16) & 31);
      const int s1 = (int)min((long long)(diag ? 17 : 32), s0 + (we - w));
      {
        const int j = bj * 32 + lane, jc = min(j, n - 1);
        __syncwarp();
        J[0][lane] = x[jc] * invL;
        J[1][lane] = y[jc] * invL;
        J[2][lane] = z[jc] * invL;
        J[3][lane] = h[jc] * invL;
        J[4][lane] = j < n ? m[jc] : 0.0;
        __syncwarp();
      }
      double bx = 0.0, by = 0.0, bz = 0.0;
#pragma unroll 1
      for (int s = s0; s < s1; ++s) {
        const int q = (lane + s) & 31;
        const double dx = xi - J[0][q], dy = yi - J[1][q];
        double dz = zi - J[2][q];
        if (KIND != kPair64R3) dz = wrap64(dz);
        double SR, SZ;
        window64<KIND>(fma(dx, dx, dy * dy), dz, hi + J[3][q], n_cut, SR, SZ);
        const bool half = diag && s == 16 && lane >= 16;  // these pairs belong to the lower lanes
        const double mj = half ? 0.0 : J[4][q], mo = half ? 0.0 : mi;
        const double mjs = mj * SR, mis = mo * SR;
        ax = fma(dx, mjs, ax);
        ay = fma(dy, mjs, ay);
        az = fma(mj, SZ, az);
        bx = fma(dx, mis, bx);
        by = fma(dy, mis, by);
        bz = fma(mo, SZ, bz);
        if (s + 1 < s1) {  // slot q + 1 comes from the lane that held it
          bx = __shfl_sync(0xffffffffu, bx, (lane + 1) & 31);
          by = __shfl_sync(0xffffffffu, by, (lane + 1) & 31);
          bz = __shfl_sync(0xffffffffu, bz, (lane + 1) & 31);
        }
      }
      const int j = bj * 32 + ((lane + s1 - 1) & 31);
      if (j < n) {
        fix64_add(F, 0, j, -bx);
        fix64_add(F, 1, j, -by);
        fix64_add(F, 2, j, -bz);
      }
      w += s1 - s0;
    }
    if (i < n) {
      fix64_add(F, 0, i, ax);
      fix64_add(F, 1, i, ay);
      fix64_add(F, 2, i, az);
    }
  }
}

}  // namespace steps
