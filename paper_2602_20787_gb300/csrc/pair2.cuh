// Two pairs per thread in packed FP32x2: the pair sums of the symmetric kernels
// (pair_sym.cuh). A thread holds two i-particles, and every quantity of its two
// pairs with one j is one 64-bit register (i0 in the lower half, i1 in the
// upper), so the whole pair is packed: separation, images, far part, envelope and
// sums. Packing the images +-k of one pair instead, as the row kernels do, leaves
// the separation, the centre image, the far ends and the sums scalar: 182 warp
// instructions per 32 pairs of the plain sum against about 100 here. Each j word
// comes from shared memory as a duplicated pair (one 128-bit load yields two
// packed operands), and one j load, one ring shuffle and one loop step serve two
// pairs.
//
// The image line is symmetric, so a pair is evaluated at |dz| and the z sum takes
// the sign of dz at the end: images |dz| - k (the near side) and |dz| + k.
#pragma once
#include <cstdint>

#include "pair_fp32.cuh"

namespace steps {

__device__ __forceinline__ u64 dup(float c) { return pk(c, c); }
__device__ __forceinline__ u64 rsq2(u64 x) {
  float a, b;
  upk(x, a, b);
  return pk(rsq(a), rsq(b));
}
__device__ __forceinline__ u64 rcp2(u64 x) {
  float a, b;
  upk(x, a, b);
  return pk(rcp_approx(a), rcp_approx(b));
}
__device__ __forceinline__ u64 max2(u64 x, float c) {
  float a, b;
  upk(x, a, b);
  return pk(fmaxf(a, c), fmaxf(b, c));
}
__device__ __forceinline__ u64 min2(u64 x, float c) {
  float a, b;
  upk(x, a, b);
  return pk(fminf(a, c), fminf(b, c));
}
constexpr u64 kSign2 = 0x8000000080000000ull;
__device__ __forceinline__ u64 abs2(u64 x) { return x & ~kSign2; }
// x with its sign flipped where s is negative
__device__ __forceinline__ u64 mulsign2(u64 x, u64 s) { return x ^ (s & kSign2); }
__device__ __forceinline__ u64 neg2(u64 x) { return x ^ kSign2; }

constexpr int kPairThreads = kBI / 2;  // threads of a block of rows: two i each

// ---- the two i-particles of a thread and a staged j-tile -------------------------
// Thread's rows of block b: 64 consecutive rows per warp, i0 and i0 + 32.
__device__ __forceinline__ int row_i0(int b) { return b * kBI + (threadIdx.x & ~31) * 2 + (threadIdx.x & 31); }

struct I2 {
  u64 xh, xl, yh, yl, zh, zl, h, m;
};

__device__ __forceinline__ I2 load_i2(const float4* __restrict__ jA, const float4* __restrict__ jB, int i0, int i1,
                                      int n) {
  const float4 a0 = jA[min(i0, n - 1)], a1 = jA[min(i1, n - 1)];
  const float4 b0 = jB[min(i0, n - 1)], b1 = jB[min(i1, n - 1)];
  // rows past n repeat the last particle with zero mass: they add nothing to the j side
  return I2{pk(a0.x, a1.x), pk(b0.x, b1.x), pk(a0.y, a1.y), pk(b0.y, b1.y), pk(a0.z, a1.z),
            pk(b0.z, b1.z), pk(b0.w, b1.w), pk(i0 < n ? a0.w : 0.0f, i1 < n ? a1.w : 0.0f)};
}

// Each word twice: XY = (x_hi, x_hi | y_hi, y_hi), XYL the lo words, Z = (z_hi | z_lo), MH = (m | h).
struct JTile2 {
  ulonglong2 XY[kBJ], XYL[kBJ], Z[kBJ], MH[kBJ];
};

// j-tile t of jt slots (slots past n: a massless particle far off the axis with zero
// softening, whose pairs are finite and add exact zeros).
template <int THREADS>
__device__ __forceinline__ void load_tile2(const float4* __restrict__ jA, const float4* __restrict__ jB, int n, int t,
                                           int jt, JTile2& T) {
  for (int s = threadIdx.x; s < jt; s += THREADS) {
    const int j = t * jt + s;
    float4 a = make_float4(4096.0f, 4096.0f, 0.0f, 0.0f), b = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (j < n) {
      a = jA[j];
      b = jB[j];
    }
    T.XY[s] = make_ulonglong2(dup(a.x), dup(a.y));
    T.XYL[s] = make_ulonglong2(dup(b.x), dup(b.y));
    T.Z[s] = make_ulonglong2(dup(a.z), dup(b.z));
    T.MH[s] = make_ulonglong2(dup(a.w), dup(b.w));
  }
}

// Kahan update of a packed sum.
template <bool KAHAN>
__device__ __forceinline__ void acc2(u64& s, u64& c, u64 v) {
  if (KAHAN) {
    const u64 y = sub2(v, c), t = add2(s, y);
    c = sub2(sub2(t, s), y);
    s = t;
  } else {
    s = add2(s, v);
  }
}
// A sum and its compensation as two doubles.
template <bool KAHAN>
__device__ __forceinline__ void sum2(u64 s, u64 c, double& a, double& b) {
  float s0, s1, c0, c1;
  upk(s, s0, s1);
  upk(c, c0, c1);
  a = (double)s0 - (KAHAN ? (double)c0 : 0.0);
  b = (double)s1 - (KAHAN ? (double)c1 : 0.0);
}

// Separation and softening sum of the two pairs, as pair_separation.
struct Sep2 {
  u64 dx, dy, dz, dr2, hh;
};
__device__ __forceinline__ void separation2(const I2& I, const JTile2& T, int q, Sep2& P) {
  const ulonglong2 xy = T.XY[q], xyl = T.XYL[q], z = T.Z[q];
  P.dx = add2(sub2(I.xh, xy.x), sub2(I.xl, xyl.x));
  P.dy = add2(sub2(I.yh, xy.y), sub2(I.yl, xyl.y));
  P.dr2 = fma2(P.dx, P.dx, mul2(P.dy, P.dy));
  const u64 d = sub2(I.zh, z.x);
  const u64 r = dup(kRound23);
  P.dz = add2(sub2(d, sub2(add2(d, r), r)), sub2(I.zl, z.y));
  P.hh = add2(I.h, T.MH[q].y);
}

// ---- near images -------------------------------------------------------------------
// One image of each pair at offset O: F / r into SR, O F / r into SZ.
__device__ __forceinline__ u64 inv_r3(u64 R2) {
  const u64 RI = rsq2(R2);
  return mul2(mul2(RI, RI), RI);
}
__device__ __forceinline__ void newton2(u64 O, u64 DR2, u64& SR, u64& SZ) {
  const u64 F = inv_r3(fma2(O, O, DR2));
  SR = add2(SR, F);
  SZ = fma2(O, F, SZ);
}
// The Newtonian images +-k.
__device__ __forceinline__ void newton_k2(u64 ADZ, float k, u64 DR2, u64& SR, u64& SZ) {
  newton2(sub2(ADZ, dup(k)), DR2, SR, SZ);
  newton2(add2(ADZ, dup(k)), DR2, SR, SZ);
}

// Softening constants of the two pairs.
struct Soft2 {
  u64 ih, nih, ih3;
};
__device__ __forceinline__ Soft2 soft2(u64 HH) {
  Soft2 s;
  s.ih = rcp2(HH);
  s.nih = neg2(s.ih);
  s.ih3 = mul2(mul2(s.ih, s.ih), s.ih);
  return s;
}
// F / r at r^2 = R2. FULL: all three branches of the spline, else u >= 1/2 on every
// lane; CENTRE: r may vanish (r^2 is floored).
template <bool FULL, bool CENTRE>
__device__ __forceinline__ u64 spline2(u64 R2, const Soft2& s) {
  const u64 RI = rsq2(CENTRE ? max2(R2, 1e-30f) : R2);
  const u64 N3 = mul2(mul2(RI, RI), RI);
  if (FULL) return spline_value_r2(R2, RI, N3, s.ih, s.nih, s.ih3);
  return spline_outer_value(mul2(R2, RI), N3, s.nih);
}
// Whether some pair of the warp has X < Y.
__device__ __forceinline__ bool any_less2(u64 X, u64 Y) {
  float xa, xb, ya, yb;
  upk(X, xa, xb);
  upk(Y, ya, yb);
  return __any_sync(0xffffffffu, xa < ya || xb < yb);
}
__device__ __forceinline__ u64 flag_nonzero2(u64 X) {  // 1 where X != 0, else 0
  float a, b;
  upk(X, a, b);
  return pk(a != 0.0f ? 1.0f : 0.0f, b != 0.0f ? 1.0f : 0.0f);
}

// The near images |k| <= M of pairs whose images k != 0 are all Newtonian, M fixed,
// in one straight run: SR, SZ the images +-1 .. +-M outward, CR the centre image's F / r
// taken as Newtonian from its R2C.
template <int M>
__device__ __forceinline__ void near_far2(u64 R2C, u64 DR2, u64 ADZ, u64& CR, u64& SR, u64& SZ) {
  CR = inv_r3(R2C);
  SR = 0;
  SZ = 0;
#pragma unroll
  for (int k = 1; k <= M; ++k) newton_k2(ADZ, (float)k, DR2, SR, SZ);
}

// Warp-uniform softening bounds of a step: kw, the largest k whose near-side image
// |dz| - k lies inside the support of some pair (k < |dz| + sqrt(h^2 - dR^2)), and k1,
// the same for the inner core u < 1/2; 0 when only centre images do.
__device__ __forceinline__ int soft_bound2(u64 H2, u64 DR2, u64 ADZ) {
  float a, b;
  upk(sub2(H2, DR2), a, b);
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"(fmaxf(a, 0.0f)));
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(b) : "f"(fmaxf(b, 0.0f)));
  // x + 2^23 - 1/2 is 2^23 + rn(x - 1/2) for x >= 1/2, and below 2^23 otherwise
  upk(add2(add2(ADZ, pk(a, b)), dup(kTwo23 - 0.5f)), a, b);
  const int k = max(__float_as_int(a), __float_as_int(b));
  return max(__reduce_max_sync(0xffffffffu, k) - kTwo23Bits, 0);
}

// The images +-k with the full spline or its outer shell.
template <bool FULL>
__device__ __forceinline__ void spline_k2(u64 ADZ, float k, u64 DR2, const Soft2& s, u64& SR, u64& SZ) {
  const u64 OA = sub2(ADZ, dup(k)), OB = add2(ADZ, dup(k));
  const u64 FA = spline2<FULL, false>(fma2(OA, OA, DR2), s), FB = spline2<FULL, false>(fma2(OB, OB, DR2), s);
  SR = add2(add2(SR, FA), FB);
  SZ = fma2(OB, FB, fma2(OA, FA, SZ));
}
__device__ __forceinline__ u64 spline_centre2(u64 R2C, u64 H2, const Soft2& s) {
  return any_less2(R2C, mul2(H2, dup(0.25f))) ? spline2<true, true>(R2C, s) : spline2<false, true>(R2C, s);
}

// The near images of a step with softened pairs: the full spline up to k1, the outer
// shell up to kw, Newtonian beyond. Every image value is the same function of (r^2, h)
// in each tier, so a pair's bits do not depend on the other lanes of its warp (in the closed
// form up to kw = kPolyMaxSoft: a step that is softened farther out takes window_walk2 for all its pairs,
// whose near range is the step's). M fixed
// (unrolled; one warp-uniform branch per k), or m at run time.
template <int M>
__device__ __forceinline__ void near_soft2(u64 DR2, const Soft2& s, u64 ADZ, int kw, int k1, u64& SR, u64& SZ) {
  SR = 0;
  SZ = 0;
#pragma unroll
  for (int k = 1; k <= M; ++k) {
    if (k > kw)
      newton_k2(ADZ, (float)k, DR2, SR, SZ);
    else if (k > k1)
      spline_k2<false>(ADZ, (float)k, DR2, s, SR, SZ);
    else
      spline_k2<true>(ADZ, (float)k, DR2, s, SR, SZ);
  }
}
// One image of each pair at offset O by the spline.
template <bool FULL>
__device__ __forceinline__ void spline_one2(u64 O, u64 DR2, const Soft2& s, u64& SR, u64& SZ) {
  const u64 F = spline2<FULL, false>(fma2(O, O, DR2), s);
  SR = add2(SR, F);
  SZ = fma2(O, F, SZ);
}
__device__ __forceinline__ void near_soft_walk2(u64 DR2, const Soft2& s, u64 ADZ, int m, int kw, int k1, u64& SR,
                                                u64& SZ) {
  SR = 0;
  SZ = 0;
  u64 TR = 0, TZ = 0;
  int k = 1;
  float fk = 1.0f;
#pragma unroll 1
  for (; k <= min(k1, m); ++k, fk += 1.0f) {
    spline_one2<true>(sub2(ADZ, dup(fk)), DR2, s, SR, SZ);
    spline_one2<true>(add2(ADZ, dup(fk)), DR2, s, TR, TZ);
  }
#pragma unroll 1
  for (; k <= min(kw, m); ++k, fk += 1.0f) {
    spline_one2<false>(sub2(ADZ, dup(fk)), DR2, s, SR, SZ);
    spline_one2<false>(add2(ADZ, dup(fk)), DR2, s, TR, TZ);
  }
#pragma unroll 2
  for (; k <= m; ++k, fk += 1.0f) {
    newton2(sub2(ADZ, dup(fk)), DR2, SR, SZ);
    newton2(add2(ADZ, dup(fk)), DR2, TR, TZ);
  }
  SR = add2(SR, TR);
  SZ = add2(SZ, TZ);
}

// The near images |k| <= m without softening, m at run time.
__device__ __forceinline__ void near_newton2(u64 R2C, u64 DR2, u64 ADZ, int m, u64& CR, u64& SR, u64& SZ) {
  CR = inv_r3(R2C);
  SR = 0;
  SZ = 0;
  u64 TR = 0, TZ = 0;  // the far side's images in sums of their own: half as many roundings on a sum
  float fk = 1.0f;
#pragma unroll 2
  for (int k = 1; k <= m; ++k, fk += 1.0f) {
    newton2(sub2(ADZ, dup(fk)), DR2, SR, SZ);
    newton2(add2(ADZ, dup(fk)), DR2, TR, TZ);
  }
  SR = add2(SR, TR);
  SZ = add2(SZ, TZ);
}

// The last image that a support of the warp's pairs can reach from |dz| <= 1/2: rn(h).
__device__ __forceinline__ int soft_reach2(u64 HH) {
  float a, b;
  upk(add2(HH, dup(kTwo23)), a, b);  // 2^23 + rn(h)
  return __reduce_max_sync(0xffffffffu, max(__float_as_int(a), __float_as_int(b))) - kTwo23Bits;
}

// What the softened images m < |k| <= kw add to a Newtonian far part: spline minus
// Newtonian. The window's edge image (k = n_cut, on one side, absent at dz = 0) ends them;
// INF (n_cut unused): over the infinite window rn(h) does, as a position that is not a number
// makes kw as large as an integer can be. (A template, so that the plain window's registers
// hold no h: at run time the choice cost 2% of its literal-law force.)
template <bool INF>
__device__ __forceinline__ void far_soft2(u64 DR2, u64 HH, const Soft2& s, u64 ADZ, int m, int kw, int n_cut, u64& SR,
                                          u64& SZ) {
  const int ke = min(kw, INF ? soft_reach2(HH) : n_cut);
  float fk = (float)(m + 1);
#pragma unroll 1
  for (int k = m + 1; k <= ke; ++k, fk += 1.0f) {
    const u64 OA = sub2(ADZ, dup(fk)), OB = add2(ADZ, dup(fk));
    const u64 RA = fma2(OA, OA, DR2), RB = fma2(OB, OB, DR2);
    u64 DA = fma2(inv_r3(RA), dup(-1.0f), spline2<true, false>(RA, s));
    u64 DB = fma2(inv_r3(RB), dup(-1.0f), spline2<true, false>(RB, s));
    if (!INF && k == n_cut) {
      DA = mul2(DA, flag_nonzero2(ADZ));
      DB = 0;
    }
    SR = add2(add2(SR, DA), DB);
    SZ = fma2(OB, DB, fma2(OA, DA, SZ));
  }
}

// ---- the far part of the line in closed form -------------------------------------
// Beyond the near images the line is a smooth function of the image number. With x the
// middle between two images, i = (x^2 + dR^2)^(-1/2), s = x i, e = i^2, the sums of
// f = 1/r^3 and z f over the images beyond x are, by the midpoint rule's
// Euler-Maclaurin series, U_R(x) = e / (1 + s) - s e^2 / 8 + ... and
// U_Z(x) = i + i e (1 - 3 s^2) / 24 + ....
//
// The two near ends lie at A +- |dz|, A = m + 1/2. Both are taken at A at once:
//   U_R(A + d) + U_R(A - d) = 2 e / (1 + s) + s e^2 T(q, d^2),
//   U_Z(A + d) - U_Z(A - d) = d s e Z(q, d^2),       q = s^2, d = |dz| <= 1/2,
// with T and Z polynomials fitted (minimax) over q in [0, 1] and d to the exact sums:
// no series is truncated. T is off by at most 8e-8 of the sum of f, Z by 5e-8 of i,
// evaluation in FP32 included. The polynomials keep the work of one side (one rsqrt,
// one rcp, 27 packed FMAs) where the series takes it twice. A = 3.5 costs least: one
// near k less saves 12 packed operations, and A = 2.5 needs 13 more coefficients.
//
// The two far ends N -+ (1/2 - |dz|) (N = n_cut) are expanded about N: one rsqrt for
// both, off by less than 6e-8 (N = 12), 1e-8 (N = 16) of terms of order one. The
// integral part 2 (N^2 - A^2) e e_N / (s + s_N) ends at N and does not cancel at large dR.
// From this n_cut on the closed form is faster than the walk of the window: at
// N = 30,000 (literal / 1:8 softening law) the walk of 20 images takes 3.95 / 2.67 ms and
// the closed form 3.43 / 2.04 ms, and from 12 on its error against FP64 is no larger than
// the walk's.
#ifndef STEPS_LINE_MIN_NCUT
#define STEPS_LINE_MIN_NCUT 12
#endif
__host__ __device__ __forceinline__ bool line_form(int n_cut) { return n_cut >= STEPS_LINE_MIN_NCUT; }
// Where every sum is compensated (the row kernels, the allocation-free call) the far ends' expansion
// shows below n_cut = 16: 2-norm error at N = 5,000, N_cut = 12 (filament) 4.98e-8 against 4.90e-8 of the
// walk, N_cut = 13 (1:8 law) 5.28e-8 against 5.22e-8, from 16 on the closed form is the better one. The
// walk takes 178 us there, the closed form 143.
__host__ __device__ __forceinline__ bool line_form_rows(int n_cut) { return n_cut >= 16; }

constexpr int kPolyNear = 3;          // m
constexpr float kPolyA = 3.5f;        // A
// Steps softened beyond this many periods take their near range up to the last
// softened image instead: the whole sum of such a pair is no longer large against the
// rounding of the Newtonian far part that its softened images would be taken from.
constexpr int kPolyMaxSoft = 8;

// The line itself.
__device__ __forceinline__ u64 line_poly_r(u64 Q, u64 D2) {
  u64 r = fma2(D2, fma2(D2, fma2(D2, dup(0.0731698186f), dup(-0.105292284f)), dup(0.0388617621f)), dup(-0.00207508531f));
  r = fma2(Q, r, dup(-5.10753242e-05f));
  r = fma2(Q, r, fma2(D2, fma2(D2, fma2(D2, dup(-0.0338161794f), dup(0.782380616f)), dup(-0.384855242f)), dup(0.0224334317f)));
  r = fma2(Q, r, fma2(D2, fma2(D2, dup(-0.319349437f), dup(0.159832034f)), dup(-0.00935625492f)));
  r = fma2(Q, r, fma2(D2, dup(2.99990705f), dup(-0.249989588f)));
  return r;
}
__device__ __forceinline__ u64 line_poly_z(u64 Q, u64 D2) {
  u64 r = fma2(D2, dup(-0.0191895589f), dup(0.0046328245f));
  r = fma2(Q, r, fma2(D2, fma2(D2, dup(-0.0732934993f), dup(0.114551534f)), dup(-0.0236126925f)));
  r = fma2(Q, r, fma2(D2, fma2(D2, dup(0.064372082f), dup(-0.104991415f)), dup(0.0218019947f)));
  r = fma2(Q, r, fma2(D2, dup(-0.388695752f), dup(0.0973390269f)));
  r = fma2(Q, r, fma2(D2, fma2(D2, dup(-0.00317250736f), dup(0.245249776f)), dup(-0.0611369641f)));
  r = fma2(Q, r, dup(-1.99999933f));
  return r;
}
// The modelled tails' n0 = 4 line: the images +-4 one by one and the continuum base of
// tail_base_fp32 beyond them (what the network or the table then corrects).
__device__ __forceinline__ u64 base_poly_r(u64 Q, u64 D2) {
  u64 r = dup(-0.0127026519f);
  r = fma2(Q, r, dup(0.0552325238f));
  r = fma2(Q, r, fma2(D2, fma2(D2, fma2(D2, dup(0.0695894838f), dup(-0.105766352f)), dup(0.0409462167f)), dup(-0.103608928f)));
  r = fma2(Q, r, dup(0.100621543f));
  r = fma2(Q, r, fma2(D2, fma2(D2, fma2(D2, dup(-0.0307293746f), dup(0.782644825f)), dup(-0.396962056f)), dup(-0.0304370083f)));
  r = fma2(Q, r, fma2(D2, fma2(D2, dup(-0.319724433f), dup(0.168626375f)), dup(-0.000903310932f)));
  r = fma2(Q, r, fma2(D2, dup(2.99861174f), dup(-0.249743871f)));
  return r;
}
__device__ __forceinline__ u64 base_poly_z(u64 Q, u64 D2) {
  u64 r = dup(0.00263720511f);
  r = fma2(Q, r, fma2(D2, dup(-0.0201418825f), dup(-0.00312730927f)));
  r = fma2(Q, r, fma2(D2, fma2(D2, dup(-0.0742022409f), dup(0.118583854f)), dup(-0.0182358385f)));
  r = fma2(Q, r, fma2(D2, fma2(D2, dup(0.0656157654f), dup(-0.108939488f)), dup(0.0256251224f)));
  r = fma2(Q, r, fma2(D2, dup(-0.387776745f), dup(0.0928691897f)));
  r = fma2(Q, r, fma2(D2, fma2(D2, dup(-0.00350156307f), dup(0.245342239f)), dup(-0.0603070125f)));
  r = fma2(Q, r, dup(-2.00002828f));
  return r;
}

// The far ends: s and e at N, and what they add to the sums to infinity (the integral
// of f ends at N). e e_N / (s + s_N): the product of the two squares leaves FP32's normal range
// from dR = 3e9 on. WIDE multiplies it and the sum by 2^60, so that it does not before the image
// sum itself, at no rounding: the row kernels, whose sums are in floating point. In the symmetric kernels all
// pairs so far apart add up to a few units of the fixed-point sums at most. (The reciprocal between the squares does
// it as well, and takes 0.9% longer in the symmetric kernels: 13.46 ms against 13.35 at N = 65,536, N_cut = 16,
// literal law.) dR^2 is finite: kPackCap.
constexpr float kFarUp = 0x1p60f;
template <bool WIDE>
__device__ __forceinline__ u64 far_rcp2(u64 x) {
  return rcp2(WIDE ? mul2(x, dup(kFarUp)) : x);
}
struct FarEnd2 {
  u64 IH, SN, EN, R, Z;
};
__device__ __forceinline__ FarEnd2 far_end2(u64 DR2, u64 ADZ, float N) {
  FarEnd2 f;
  f.IH = rsq2(add2(DR2, dup(N * N)));
  f.SN = mul2(f.IH, dup(N));
  f.EN = mul2(f.IH, f.IH);
  const u64 D = sub2(ADZ, dup(0.5f)), D2 = mul2(D, D);
  const u64 G = mul2(f.SN, f.EN);
  const u64 ZN = fma2(mul2(f.EN, fma2(mul2(f.SN, f.SN), dup(-15.0f), dup(9.0f))),
                      fma2(D2, dup(-1.0f / 3.0f), dup(1.0f / 12.0f)), dup(2.0f));
  f.R = mul2(mul2(G, f.EN), fma2(D2, dup(-3.0f), dup(0.25f)));
  f.Z = mul2(mul2(D, G), ZN);
  return f;
}
// At dz = 0 the window has no edge image and the z sum vanishes (the images' fused
// products leave a rounding). EDGE: the sums hold the edge image.
template <bool EDGE>
__device__ __forceinline__ void fix_dz0(u64 ADZ, u64 DR2, float N, u64& SR, u64& SZ) {
  float za, zb;
  upk(ADZ, za, zb);
  if (fminf(za, zb) == 0.0f) {
    float ea, eb, ra, rb, sa, sb;
    if (EDGE) {
      upk(inv_r3(add2(DR2, dup(N * N))), ea, eb);
      upk(SR, ra, rb);
      SR = pk(za == 0.0f ? ra - ea : ra, zb == 0.0f ? rb - eb : rb);
    }
    upk(SZ, sa, sb);
    SZ = pk(za == 0.0f ? 0.0f : sa, zb == 0.0f ? 0.0f : sb);
  }
}

// The images beyond the near ones |k| <= kPolyNear added to (SR, SZ), at ADZ >= 0. INF:
// the infinite line, else the window of N. BASE: with the modelled tails' base.
template <bool INF, bool BASE, bool WIDE = false>
__device__ __forceinline__ void line_far2(u64 DR2, u64 ADZ, float N, u64& SR, u64& SZ) {
  const u64 IL = rsq2(add2(DR2, dup(kPolyA * kPolyA)));
  const u64 S = mul2(IL, dup(kPolyA)), E = mul2(IL, IL);
  const u64 Q = mul2(S, S), D2 = mul2(ADZ, ADZ), G = mul2(S, E);
  const u64 T = BASE ? base_poly_r(Q, D2) : line_poly_r(Q, D2);
  const u64 Z = BASE ? base_poly_z(Q, D2) : line_poly_z(Q, D2);
  u64 I;
  if (INF) {
    I = mul2(mul2(E, dup(2.0f)), rcp2(add2(S, dup(1.0f))));
  } else {
    const FarEnd2 f = far_end2(DR2, ADZ, N);
    constexpr float UP = WIDE ? kFarUp : 1.0f;
    const u64 EE = mul2(mul2(E, dup(2.0f * UP * (N * N - kPolyA * kPolyA))), f.EN);
    I = fma2(EE, far_rcp2<WIDE>(add2(S, f.SN)), f.R);
    SZ = add2(SZ, f.Z);
  }
  SR = add2(SR, fma2(mul2(G, E), T, I));
  SZ = fma2(mul2(ADZ, G), Z, SZ);
}

// One side of the line beyond any x = LO >= 4: minus the sum of f, its integral ending
// at N, and the sum of z f to infinity less its integral IL. The Euler-Maclaurin series'
// first three corrections, with coefficients (beyond the first) fitted over x >= 4:
// off by at most 1.1e-7 and 4e-8 of themselves.
struct LineSide2 {
  u64 NR, IL, Z;
};
template <bool WIDE>
__device__ __forceinline__ LineSide2 line_side2(u64 LO, u64 DR2, const FarEnd2& f, float N2) {
  const u64 IL = rsq2(fma2(LO, LO, DR2));
  const u64 S = mul2(LO, IL), E = mul2(IL, IL);
  const u64 EE = mul2(WIDE ? mul2(E, dup(kFarUp)) : E, f.EN);
  const u64 NI = mul2(mul2(fma2(LO, LO, dup(-N2)), EE), far_rcp2<WIDE>(add2(S, f.SN)));
  const u64 Q = mul2(S, S), W = mul2(E, Q);
  u64 PR = fma2(W, dup(0.238131417f), fma2(E, dup(-0.168406769f), dup(-0.127495596f)));
  PR = fma2(W, PR, fma2(E, dup(0.0547808694f), dup(0.125f)));
  u64 PZ = fma2(W, fma2(Q, dup(-0.18554619f), dup(0.166497663f)), fma2(Q, dup(0.127402248f), dup(-0.107906074f)));
  PZ = fma2(W, PZ, fma2(E, dup(0.00946691296f), fma2(Q, dup(-0.125010776f), dup(0.0416820926f))));
  return LineSide2{fma2(mul2(mul2(E, E), S), PR, NI), IL, mul2(mul2(IL, E), PZ)};
}

// ---- image sums of the plain window ------------------------------------------------
// The images one by one up to m (softened: to the bounds kw, k1), then the far part of
// each side in closed form from A = m + 1/2, or for m = n_cut - 1 the edge image.
template <bool WIDE>
__device__ __forceinline__ void window_walk2(u64 DR2, u64 HH, u64 R2C, u64 ADZ, bool soft, int m, int n_cut,
                                             float fnc, u64& SR, u64& SZ) {
  u64 CR, H2 = mul2(HH, HH);
  int kw = -1;
  if (soft) {
    const Soft2 s = soft2(HH);
    kw = soft_bound2(H2, DR2, ADZ);
    m = min(max(m, kw), n_cut - 1);
    CR = spline_centre2(R2C, H2, s);
    near_soft_walk2(DR2, s, ADZ, m, kw, soft_bound2(mul2(H2, dup(0.25f)), DR2, ADZ), SR, SZ);
  } else {
    near_newton2(R2C, DR2, ADZ, m, CR, SR, SZ);
  }
  SR = add2(SR, CR);
  SZ = fma2(ADZ, CR, SZ);
  if (m == n_cut - 1) {
    const u64 OE = sub2(ADZ, dup(fnc)), RE = fma2(OE, OE, DR2);
    const u64 FE = mul2(kw >= n_cut ? spline2<true, false>(RE, soft2(HH)) : inv_r3(RE), flag_nonzero2(ADZ));
    SR = add2(SR, FE);
    SZ = fma2(OE, FE, SZ);
    fix_dz0<false>(ADZ, DR2, fnc, SR, SZ);
    return;
  }
  const FarEnd2 f = far_end2(DR2, ADZ, fnc);
  const float A = (float)m + 0.5f;
  const LineSide2 a = line_side2<WIDE>(add2(ADZ, dup(A)), DR2, f, fnc * fnc);
  const LineSide2 b = line_side2<WIDE>(sub2(dup(A), ADZ), DR2, f, fnc * fnc);
  SR = add2(SR, sub2(f.R, add2(a.NR, b.NR)));
  // the integrals of z f, IL_a - IL_b, without cancellation at large dR
  const u64 P = mul2(a.IL, b.IL);
  const u64 PP = mul2(WIDE ? mul2(P, dup(kFarUp)) : P, P);
  const u64 IZ = mul2(mul2(PP, mul2(ADZ, dup(-4.0f * A))), far_rcp2<WIDE>(add2(a.IL, b.IL)));
  SZ = add2(SZ, add2(add2(IZ, sub2(a.Z, b.Z)), f.Z));
  fix_dz0<true>(ADZ, DR2, fnc, SR, SZ);
}
// The same out of line, for the rare steps of the closed form.
template <bool WIDE>
static __device__ __noinline__ ulonglong2 window_walk_call2(u64 DR2, u64 HH, u64 ADZ, int n_cut) {
  u64 SR, SZ;
  window_walk2<WIDE>(DR2, HH, fma2(ADZ, ADZ, DR2), ADZ, true, kPolyMaxSoft, n_cut, (float)n_cut, SR, SZ);
  return make_ulonglong2(SR, SZ);
}

// SR = sum F / r, SZ = sum o F / r over the window of n_cut. LINE: the images beyond
// the near ones in closed form (line_form(n_cut)), else every image walked.
// FAR: every h_i + h_j below half a period, so only the centre image can be
// softened: the near images are taken as Newtonian in one straight run and the centre
// replaced where it is softened. WIDE: see far_end2.
template <bool LINE, bool FAR, bool WIDE = false>
__device__ __forceinline__ void window2(const Sep2& P, int n_cut, float fnc, u64& SR, u64& SZ) {
  static_assert(!FAR || LINE, "the straight run belongs to the closed far part");
  const u64 ADZ = abs2(P.dz);
  const u64 R2C = fma2(ADZ, ADZ, P.dr2), H2 = mul2(P.hh, P.hh);
  const bool soft = any_less2(R2C, H2);
  if (!LINE) {
    window_walk2<WIDE>(P.dr2, P.hh, R2C, ADZ, soft, n_cut - 1, n_cut, fnc, SR, SZ);
    SZ = mulsign2(SZ, P.dz);
    return;
  }
  u64 CR;
  if (FAR || !soft) near_far2<kPolyNear>(R2C, P.dr2, ADZ, CR, SR, SZ);
  if (soft) {
    const Soft2 s = soft2(P.hh);
    if (FAR) {
      CR = spline2<true, true>(R2C, s);
    } else {
      const int kw = soft_bound2(H2, P.dr2, ADZ);
      if (kw > kPolyMaxSoft) {
        const ulonglong2 w = window_walk_call2<WIDE>(P.dr2, P.hh, ADZ, n_cut);
        SR = w.x;
        SZ = mulsign2(w.y, P.dz);
        return;
      }
      CR = spline_centre2(R2C, H2, s);
      near_soft2<kPolyNear>(P.dr2, s, ADZ, kw, soft_bound2(mul2(H2, dup(0.25f)), P.dr2, ADZ), SR, SZ);
      if (kw > kPolyNear) far_soft2<false>(P.dr2, P.hh, s, ADZ, kPolyNear, kw, n_cut, SR, SZ);
    }
  }
  SR = add2(SR, CR);
  SZ = fma2(ADZ, CR, SZ);
  line_far2<false, false, WIDE>(P.dr2, ADZ, fnc, SR, SZ);
  fix_dz0<true>(ADZ, P.dr2, fnc, SR, SZ);
  SZ = mulsign2(SZ, P.dz);
}

// ---- the row kernel of the plain window -----------------------------------------
// Rows against every j (shards' row step, loads whose sums fixed point does not resolve): the
// work split and partial layout of the row kernels, [slot][3][kBI] doubles, slot = i-block + CTA. The
// units cover the i-blocks [b0, b0 + U / NT), and slots count i-blocks from b0. A unit's j-tile has jt slots, 128
// or fewer where that lets the places for CTAs share the units more evenly: the time goes as the largest number of units
// of a place times jt and some 14 more for the tile's staging (N = 10,000, N_cut = 8 .. 16: 507 / 557 us whole / in
// quarters; N = 2,000, N_cut = 8: 75 / 56).
#ifndef STEPS_ROW_MIN_BLOCKS
#define STEPS_ROW_MIN_BLOCKS 10  // resident CTAs per SM the kernel is compiled for (registers)
#endif
struct RowSplit {
  long long U;
  int NT, jt, C;
};
// The most CTAs that row_split gives any number of blocks up to `blocks` (partials are allocated for them).
inline int row_ctas(int blocks, int n, int ctas) {
  const long long U = (long long)blocks * ((n + 31) / 32);
  return (int)(U < ctas ? U : ctas);
}
inline RowSplit row_split(int blocks, int n, int ctas) {
  const int places = ctas < 152 * STEPS_ROW_MIN_BLOCKS ? ctas : 152 * STEPS_ROW_MIN_BLOCKS;
  RowSplit best{0, 0, 0, 0};
  long long cost = 0;
  for (int jt = kBJ; jt >= 32; jt /= 2) {
    const int NT = (n + jt - 1) / jt;
    const long long U = (long long)blocks * NT;
    const int C = (int)(U < ctas ? U : ctas);
    const long long t = (U + places - 1) / places * (jt + 14);
    if (best.jt == 0 || t < cost) {
      best = RowSplit{U, NT, jt, C};
      cost = t;
    }
  }
  return best;
}
template <bool KAHAN, bool LINE>
__global__ void __launch_bounds__(kPairThreads, STEPS_ROW_MIN_BLOCKS)
pair_row_kernel(const float4* __restrict__ jA, const float4* __restrict__ jB, int n, int n_cut, long long U, int NT,
                int jt, int C, double* __restrict__ part, int b0, const int* __restrict__ skip = nullptr) {
  __shared__ JTile2 T;
  if (skip && *skip) return;  // the symmetric kernel has taken the pairs
  const int c = blockIdx.x;
  const long long u1 = (long long)(c + 1) * U / C;
  const float fnc = (float)n_cut;
  long long u = (long long)c * U / C;
  while (u < u1) {
    const int lb = (int)(u / NT);  // i-block of the evaluated range
    const int t0 = (int)(u % NT);
    const int t1 = (int)min((long long)NT, (long long)t0 + (u1 - u));
    const int i0 = row_i0(b0 + lb);
    const I2 I = load_i2(jA, jB, i0, i0 + 32, n);
    u64 sx = 0, sy = 0, sz = 0, cx = 0, cy = 0, cz = 0;
    for (int t = t0; t < t1; ++t) {
      __syncthreads();
      load_tile2<kPairThreads>(jA, jB, n, t, jt, T);
      __syncthreads();
#pragma unroll 1
      for (int k0 = 0; k0 < jt; k0 += STEPS_KAHAN_GROUP) {
        u64 gx = 0, gy = 0, gz = 0;
#pragma unroll 1
        for (int k = k0; k < k0 + STEPS_KAHAN_GROUP; ++k) {
          Sep2 P;
          separation2(I, T, k, P);
          u64 SR, SZ;
          window2<LINE, false, true>(P, n_cut, fnc, SR, SZ);
          const u64 m = T.MH[k].x, MS = mul2(m, SR);
          gx = fma2(P.dx, MS, gx);
          gy = fma2(P.dy, MS, gy);
          gz = fma2(m, SZ, gz);
        }
        acc2<KAHAN>(sx, cx, gx);
        acc2<KAHAN>(sy, cy, gy);
        acc2<KAHAN>(sz, cz, gz);
      }
    }
    double* dst = part + ((long long)lb + c) * 3 * kBI + (i0 - (b0 + lb) * kBI);
    sum2<KAHAN>(sx, cx, dst[0], dst[32]);
    sum2<KAHAN>(sy, cy, dst[kBI], dst[kBI + 32]);
    sum2<KAHAN>(sz, cz, dst[2 * kBI], dst[2 * kBI + 32]);
    u += t1 - t0;
  }
}

}  // namespace steps
