// Symmetric evaluation of the pair sum (Newton's third law). The window of
// eq. ForceCylindrical is symmetric: the reverse pair (j, i) sees the images of
// (i, j) mirrored, with the same dR and h_i + h_j, so its sums are sr(j, i) =
// sr(i, j) and sz(j, i) = -sz(i, j), and the force j feels from i is the
// opposite of the force i feels from j up to the two masses. Each unordered
// pair is therefore evaluated once: with v = (dx sr, dy sr, sz),
//   S_i += m_j v,   S_j -= m_i v,
// where S is the sum that the FP32 pair kernels produce per particle (scaled by
// -G / L^2 in the finalize step).
//
// Work split. The (i-block b, j-tile t) units of the upper triangle of the block
// grid are laid out b-major, and every CTA takes an equal contiguous range, as in the
// stream-K split of the row kernels. A block is 128 rows, two per thread (pair2.cuh),
// so a CTA is two warps. A tile is a block's 128 rows, or a quarter of them when there
// are too few blocks to fill the GPU: at N = 2,048 the 136 whole units leave most SMs one
// CTA (134 us a force), the 544 quarter units take 55 us, their steps split in two 50. A unit of the diagonal block evaluates
// all ordered pairs for the i side only (the self pair adds exact zeros); the others
// evaluate their pairs once and add each to both sides.
//
// The j side. In each group of 32 j-slots of a tile, lane l pairs its two i with
// slot (l + s) mod 32 at step s, so every slot meets every lane once in 32
// steps. A lane keeps the running sum of m_i v for the slot it holds and passes
// it to lane l - 1 after each step (JRing: one shuffle per component and step).
// After the tile, thread q adds the two warps' sums of j-slot q.
//
// Accumulation. The i-side sum of a CTA's range (FP32, Kahan-compensated as in
// the row kernels) and the j-side sum of a unit are converted to 64-bit fixed
// point, value * 2^S rounded to an integer, and added with integer atomics into
// one accumulator per particle and component. Integer addition is associative,
// so the result does not depend on the order in which CTAs finish: the force
// evaluation stays deterministic and bit-reproducible. 2^S is chosen on the host
// from a bound on |S_i| (total mass times the largest softened force); a value
// beyond 2^62 / 2^S sets an error bit instead of wrapping. The R^3 force, the allocation-free
// call and the FP64 form (pair_fp64.cuh) take two words per sum: see "Scale and spread" below.
#pragma once
#include <cstdint>

#include "pair2.cuh"
#include "surrogate_pair.cuh"
#include "tail_table.cuh"

namespace steps {

constexpr int kErrFixRange = 32;  // a pair sum left the range of the fixed-point accumulators
constexpr int kMaxFixExpF = 120;  // the largest scale exponent taken as a float
constexpr int kErrIndex = 64;     // (index-checked builds) an index left its buffer

// Index-checked builds (STEPS_DEBUG_INDEX=1) check every computed index of the
// symmetric kernels' shared and global accesses against its buffer; an index
// outside is recorded in g_index_err and clamped into the buffer, so that
// control flow (and every warp-collective call) stays the same. The host folds
// the record into the device error word (kErrIndex). Release builds compile
// the checks away.
#ifndef STEPS_DEBUG_INDEX
#define STEPS_DEBUG_INDEX 0
#endif
#if STEPS_DEBUG_INDEX
__device__ unsigned int g_index_err;
#endif

__device__ __forceinline__ long long checked_index(long long v, long long size) {
#if STEPS_DEBUG_INDEX
  if (v < 0 || v >= size) {
    atomicOr(&g_index_err, 1u);
    return v < 0 ? 0 : size - 1;
  }
#else
  (void)size;
#endif
  return v;
}
constexpr int kJRow = 3 * kBJ;    // floats of one warp's j-side row: [kBJ][3]
constexpr int kSymThreads = kPairThreads;

// Resident CTAs (of two warps) per SM the kernels are compiled for, i.e. their
// registers. Measured at N = 65,536, N_cut = 64 (1:8 / literal law): plain 9.62 / 16.4 ms at
// 8, 9.67 / 15.9 at 10, 9.76 / 15.9 at 12, so the straight run takes 8 and the tiered form
// 10; table 11.7 / 17.6, 11.8 / 17.5, 11.4 / 17.5; network 23.3 / 30.7 at 6, 23.4 / 29.6 at 7 and 8.
#ifndef STEPS_SYM_FAR_MIN_BLOCKS
#define STEPS_SYM_FAR_MIN_BLOCKS 8
#endif
#ifndef STEPS_SYM_MIN_BLOCKS
#define STEPS_SYM_MIN_BLOCKS 10
#endif
#ifndef STEPS_SYM_SURR_MIN_BLOCKS
#define STEPS_SYM_SURR_MIN_BLOCKS 7
#endif
#ifndef STEPS_SYM_TABLE_MIN_BLOCKS
#define STEPS_SYM_TABLE_MIN_BLOCKS 12
#endif

// Fixed-point accumulators (two's complement in unsigned words, unit
// 1 / scale) and the error word. Unsharded (world == 0): acc[3][n]. When the
// rows are sharded across world ranks (balanced contiguous ranges of 128-row
// blocks: the first `extra` ranks own base + 1 blocks, the others base),
// acc[world][3][chunk], rank-major, so that a reduce-scatter over the ranks
// hands each rank the sums of its own rows.
struct FixAcc {
  unsigned long long* acc;
  int n;
  double scale;
  float scale_f;  // the scale when it is a normal float, else 0
  int* err;
  int world, base, extra, chunk;
  unsigned long long* lo = nullptr;  // low words [3][n] of two-word sums (unsharded)
};

// Scale and spread. With B a bound on any |S_i| the scale is 2^57 / B, so one unit is 2^-57 B,
// and how that compares with the sums themselves is a matter of the load: B holds the force at
// the smallest softening, a typical sum the force at the distances between the particles. A
// sum of two words (hi in units of 1 / scale, lo the remainder in units of 2^-kLoBits / scale)
// resolves 2^-97 B. The spread is B over an estimate from below of a typical sum: the mass
// beside the heaviest particle at the load's largest separation D (units of L), in R^3 over D^2
// and in the cylinder over the line's D sqrt(N^2 + D^2) / (2 N), N = n_cut. It has no units: it is the
// same for any total mass and, in R^3, any unit of length. Up to kMaxSpread the unit is 2^-69 of a
// typical sum, below FP64's rounding also when a load spreads a hundredfold between two looks at it: for
// contexts (a softening of some 1e-4 of the load's size; their row kernels are as fast in R^3). The
// allocation-free call looks at every load and adds FP32 sums: up to kMaxSpreadF, 2^-45 (1e-8 of the size).
// Beyond, the row kernels take the pairs.
constexpr int kLoBits = 40;
constexpr double kMaxSpread = 0x1p28, kMaxSpreadF = 0x1p52;

// B: one image's softened force is at most 4 / hh^2 <= (L / h_min)^2 = q^2 (the peak of the
// spline of eq. Force_spline_kernel with hh >= 2 h_min), the other images of the window add at
// most 2 sum_k 1 / (k - 1/2)^2 < 10 (none in R^3), and the masses add up to M.
__host__ __device__ __forceinline__ double fix_bound(double M, double q, bool images) {
  return M * (q * q + (images ? 10.0 : 0.0));
}
// Whether the spread is at most `most` (n_cut = 0: R^3), without a division or a root: sqrt(N^2 + D^2)
// is taken as N + D.
__host__ __device__ __forceinline__ bool fix_resolves(double B, double M, double m_max, double D, int n_cut, double most) {
  const double N = n_cut, T = most * (M - m_max);
  return n_cut > 0 ? B * D * (N + D) <= 2.0 * N * T : B * D * D <= T;
}

__device__ __forceinline__ long long fix_index(const FixAcc& F, int c, int i) {
  if (F.world == 0) return (long long)c * F.n + i;
  const int b = i / kBI, big = F.extra * (F.base + 1);
  const int r = b < big ? b / (F.base + 1) : F.extra + (b - big) / F.base;
  const int first = (r < F.extra ? r * (F.base + 1) : big + (r - F.extra) * F.base) * kBI;
  return ((long long)r * 3 + c) * F.chunk + (i - first);
}

// value * scale as a 64-bit integer (and, TWO, the remainder); one beyond 2^62 (or not finite)
// sets the error bit and gives 0, so that nothing ever wraps. The scale is a power of two: where it
// is a normal float (F.scale_f, else 0) the product is exact in FP32 and the conversion keeps
// off the FP64 pipe, whose 2 lanes per SM and clock took 10 of the 40 us of an R^3
// force at N = 5,000 (three or four FP64 operations per sum).
struct FixValue {
  long long hi, lo;
  __device__ __forceinline__ void add(const FixValue& v) {
    hi += v.hi;
    lo += v.lo;
  }
  __device__ __forceinline__ void sub(const FixValue& v) {
    hi -= v.hi;
    lo -= v.lo;
  }
};
template <bool TWO>
__device__ __forceinline__ FixValue fix_value(const FixAcc& F, float v) {
  if (F.scale_f > 0.0f) {
    const float q = v * F.scale_f;
    if (fabsf(q) < 4.0e18f)
      return {__float2ll_rn(q), TWO ? __float2ll_rn((q - rintf(q)) * (float)(1LL << kLoBits)) : 0};
  } else {
    const double q = (double)v * F.scale;
    if (fabs(q) < 4.0e18)
      return {__double2ll_rn(q), TWO ? __double2ll_rn((q - rint(q)) * (double)(1LL << kLoBits)) : 0};
  }
  atomicOr(F.err, kErrFixRange);
  return {0, 0};
}
template <bool TWO>
__device__ __forceinline__ void fix_add(const FixAcc& F, int c, int i, const FixValue& q) {
  const long long size = F.world == 0 ? 3LL * F.n : 3LL * F.world * F.chunk;
  const long long o = checked_index(fix_index(F, c, i), size);
  atomicAdd(F.acc + o, (unsigned long long)q.hi);
  if (TWO) atomicAdd(F.lo + o, (unsigned long long)q.lo);
}
// The sums of rows i0 and i1 (packed s, compensation k) into component c.
template <bool KAHAN, bool TWO>
__device__ __forceinline__ void fix_add_rows(const FixAcc& F, int c, int i0, int i1, u64 s, u64 k) {
  float s0, s1, k0, k1;
  upk(s, s0, s1);
  upk(k, k0, k1);
  FixValue v0 = fix_value<TWO>(F, s0), v1 = fix_value<TWO>(F, s1);
  if (KAHAN) {
    v0.sub(fix_value<TWO>(F, k0));
    v1.sub(fix_value<TWO>(F, k1));
  }
  if (i0 < F.n) fix_add<TWO>(F, c, i0, v0);
  if (i1 < F.n) fix_add<TWO>(F, c, i1, v1);
}

// Offset of row b of the upper triangle (units t = b .. NB - 1 per row).
__host__ __device__ __forceinline__ long long tri_off(int b, int NB) {
  return (long long)b * NB - (long long)b * (b - 1) / 2;
}

// The row b of unit u (tri_off(b) <= u < tri_off(b + 1)).
__device__ __forceinline__ int tri_row(long long u, int NB) {
  const double h = 2.0 * NB + 1.0;
  int b = (int)(0.5 * (h - sqrt(fmax(h * h - 8.0 * (double)u, 0.0))));
  b = max(0, min(b, NB - 1));
  while (b > 0 && tri_off(b, NB) > u) --b;
  while (b + 1 < NB && tri_off(b + 1, NB) <= u) ++b;
  return b;
}

// The j-slot that this lane pairs with at step k of a tile: in each group of 32
// slots lane l takes slot (l + k) mod 32, so every slot meets every lane once.
__device__ __forceinline__ int jslot(int k) {
  return (int)checked_index((k & ~31) | ((k + (int)threadIdx.x) & 31), kBJ);
}

// The j side carried around the warp: a lane keeps the running sum of the slot it
// holds, adds both its pairs' vectors, and takes over the sum of lane l + 1 (the
// slot it holds at the next step): one shuffle per component and step for 64 pairs.
// After each group of STEPS_KAHAN_GROUP steps the sums (of 2 x 8 terms) are added
// to the slots' sums in the warp's shared row, so that no FP32 running sum is
// longer than those groups.
// COMP: after every kCompGroup steps, and the rounding of each sum of groups is kept beside it (exactly, by
// the two-sum), in the second half of a row of 2 kJRow floats, so that only the groups themselves round, as on the
// i side. The R^3 force and the allocation-free call under Kahan summation take it, whose rows had a
// compensated sum over every j before: 2-norm error against FP64 over ten loads, rows / without it / with it, R^3 at
// N = 20,000 3.37e-7 / 3.38e-7 / 3.34e-7 (2.3% of its time beside groups of 8 steps), the call at N = 10,007, N_cut = 16
// 3.944e-8 / 3.989e-8 / 3.942e-8 (4% of its time).
constexpr int kCompGroup = 4;
template <bool COMP>
struct JRing {
  float a[3] = {0.f, 0.f, 0.f};
  // a += m_i v of both pairs: M = m_i, X = m_i sr (packed); COMP: z fused, as on the i side
  __device__ __forceinline__ void take(u64 DX, u64 DY, u64 M, u64 X, u64 SZ, bool shift_on) {
    float x0, x1, d0, d1, z0, z1;
    upk(X, x0, x1);
    upk(DX, d0, d1);
    a[0] = fmaf(d1, x1, fmaf(d0, x0, a[0]));
    upk(DY, d0, d1);
    a[1] = fmaf(d1, x1, fmaf(d0, x0, a[1]));
    if (COMP) {
      upk(M, d0, d1);
      upk(SZ, z0, z1);
      a[2] = fmaf(d1, z1, fmaf(d0, z0, a[2]));
    } else {
      upk(mul2(M, SZ), z0, z1);
      a[2] += z0 + z1;
    }
    if (shift_on) shift();
  }
  // a += both halves of V
  __device__ __forceinline__ void add(const u64 (&V)[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float v0, v1;
      upk(V[c], v0, v1);
      a[c] += v0 + v1;
    }
  }
  __device__ __forceinline__ void shift() {
#pragma unroll
    for (int c = 0; c < 3; ++c) a[c] = __shfl_sync(0xffffffffu, a[c], (threadIdx.x + 1) & 31);
  }
  // k: the group's last step; first: the first group of its 32 slots
  __device__ __forceinline__ void flush(float* row, int k, bool first) {
    float* d = row + 3 * jslot(k);
    __syncwarp();  // the slots' last sums were written by other lanes
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (!COMP) {
        d[c] = first ? a[c] : d[c] + a[c];
      } else if (first) {
        d[c] = a[c];
        d[kJRow + c] = 0.f;
      } else {
        const float o = d[c], t = o + a[c], b = t - o;
        d[kJRow + c] += (o - (t - b)) + (a[c] - b);
        d[c] = t;
      }
      a[c] = 0.f;
    }
  }
};
static_assert(32 % STEPS_KAHAN_GROUP == 0 && STEPS_KAHAN_GROUP % kCompGroup == 0, "a round of 32 slots holds whole groups");

// ---- pair forms ------------------------------------------------------------------
// A form gives the image sums (SR, SZ) of a thread's two pairs.

// The plain window (pair2.cuh).
template <bool LINE, bool FAR>
struct PlainForm {
  int n_cut;
  float fnc;
  __device__ __forceinline__ void operator()(const Sep2& P, u64& SR, u64& SZ) const {
    window2<LINE, FAR>(P, n_cut, fnc, SR, SZ);
  }
};

// How the modelled tails' near images and base are taken:
//   kModelWide4, kModelInf4: n0 = 4 in closed form (line_far2), the window's far ends
//     expanded about n_cut (n_cut >= kWideNcut) or at infinity;
//   kModelExact, kModelInf: any n0, near images walked, the base of tail_base_fp32
//     side by side with each far end on its own, or at infinity.
enum Model { kModelWide4, kModelInf4, kModelExact, kModelInf };
// From this n_cut on the expansion's error in the base is below 2e-9 (its first
// dropped term is 60 / n_cut^6 times at most 0.0052).
constexpr int kWideNcut = 24;
__host__ __device__ constexpr bool model_inf(int m) { return m == kModelInf4 || m == kModelInf; }
__host__ __device__ constexpr bool model_poly(int m) { return m == kModelWide4 || m == kModelInf4; }

// One side of the base of tail_base_fp32, x = LO: the sums with the first
// Euler-Maclaurin term of the near end. The integral of f ends at the far end with
// s, e = SE, EE there and NUM the difference of the squared ends (INF: at infinity).
template <bool INF>
__device__ __forceinline__ void base_side2(u64 LO, u64 DR2, u64 SE, u64 EE, u64 NUM, u64& R, u64& Z) {
  const u64 IL = rsq2(fma2(LO, LO, DR2));
  const u64 E = mul2(IL, IL), S = mul2(LO, IL);
  u64 I = mul2(E, rcp2(add2(S, SE)));
  if (!INF) I = mul2(I, mul2(EE, NUM));
  R = fma2(mul2(mul2(E, E), S), dup(-0.125f), I);
  Z = fma2(mul2(IL, E), fma2(mul2(S, S), dup(-0.125f), dup(1.0f / 24.0f)), IL);
}

// The base for any n0 and each far end on its own, added to (SR, SZ).
template <bool INF>
__device__ __forceinline__ void base2(u64 DR2, u64 ADZ, const SurrConst& S, u64& SR, u64& SZ) {
  const u64 LA = add2(ADZ, dup(S.A)), LB = sub2(dup(S.A), ADZ);
  u64 RA, ZA, RB, ZB;
  if (INF) {
    base_side2<INF>(LA, DR2, dup(1.0f), 0, 0, RA, ZA);
    base_side2<INF>(LB, DR2, dup(1.0f), 0, 0, RB, ZB);
  } else {
    // + side: n_cut - 1/2 + |dz|; - side: n_cut + 1/2 - |dz| when dz != 0 (the edge image belongs to it)
    const u64 HA = add2(ADZ, dup(S.fnh));
    const u64 HB = sub2(add2(dup(S.fnh), flag_nonzero2(ADZ)), ADZ);
    const u64 IA = rsq2(fma2(HA, HA, DR2)), IB = rsq2(fma2(HB, HB, DR2));
    const u64 EA = mul2(IA, IA), EB = mul2(IB, IB), TA = mul2(HA, IA), TB = mul2(HB, IB);
    base_side2<INF>(LA, DR2, TA, EA, mul2(sub2(HA, LA), add2(HA, LA)), RA, ZA);
    base_side2<INF>(LB, DR2, TB, EB, mul2(sub2(HB, LB), add2(HB, LB)), RB, ZB);
    SR = fma2(add2(mul2(mul2(EA, EA), TA), mul2(mul2(EB, EB), TB)), dup(0.125f), SR);
    const u64 FA = fma2(mul2(IA, EA), fma2(mul2(TA, TA), dup(-0.125f), dup(1.0f / 24.0f)), IA);
    const u64 FB = fma2(mul2(IB, EB), fma2(mul2(TB, TB), dup(-0.125f), dup(1.0f / 24.0f)), IB);
    SZ = add2(SZ, sub2(FB, FA));
  }
  SR = add2(SR, add2(RA, RB));
  SZ = add2(SZ, sub2(ZA, ZB));
}

// State of a modelled tail's pair across the network or the table read: the image
// sums are a0 + b0 y0 and a1 + b1 y1 in the model's outputs; u: its inputs.
struct Model2 {
  u64 a0, b0, a1, b1;
  u64 u[3];
};

// Near images, base, envelope and inputs of a modelled tail (see surr_stage_a), with
// the exact spline in place of softened images of the tail. RAW: no base and unit
// envelope (the nearest-image table).
template <int MODEL, bool RAW, bool FAR>
__device__ __forceinline__ void model_stage2(const Sep2& P, u64 ADZ, int n_cut, const SurrConst& S, Model2& M) {
  constexpr bool POLY = model_poly(MODEL), INF = model_inf(MODEL);
  static_assert(!FAR || POLY, "the straight run belongs to the closed near part");
  const u64 dR = mul2(P.dr2, rsq2(max2(P.dr2, 1e-30f)));
  M.u[0] = fma2(min2(dR, S.dR_max), dup(S.two_inv_dR_max), dup(-1.0f));
  M.u[1] = fma2(ADZ, dup(4.0f), dup(-1.0f));
  M.u[2] = fma2(min2(P.hh, S.A), dup(S.two_over_A), dup(-1.0f));
  const int m = POLY ? kPolyNear : S.n0;
  const u64 R2C = fma2(ADZ, ADZ, P.dr2);
  u64 CR, SR, SZ;
  const u64 H2 = mul2(P.hh, P.hh);
  const bool soft = any_less2(R2C, H2);
  if (FAR || (POLY && !soft)) near_far2<kPolyNear>(R2C, P.dr2, ADZ, CR, SR, SZ);
  if (soft) {
    const Soft2 s = soft2(P.hh);
    if (FAR) {
      CR = spline2<true, true>(R2C, s);
    } else {
      const int kw = soft_bound2(H2, P.dr2, ADZ), k1 = soft_bound2(mul2(H2, dup(0.25f)), P.dr2, ADZ);
      CR = spline_centre2(R2C, H2, s);
      if (POLY)
        near_soft2<kPolyNear>(P.dr2, s, ADZ, kw, k1, SR, SZ);
      else
        near_soft_walk2(P.dr2, s, ADZ, m, kw, k1, SR, SZ);
      if (kw > m) far_soft2<INF>(P.dr2, P.hh, s, ADZ, m, kw, n_cut, SR, SZ);
    }
  } else if (!POLY) {
    near_newton2(R2C, P.dr2, ADZ, m, CR, SR, SZ);
  }
  SR = add2(SR, CR);
  SZ = fma2(ADZ, CR, SZ);
  if (RAW) {
    M.a0 = SR;
    M.a1 = SZ;
    M.b0 = M.b1 = dup(1.0f);
    return;
  }
  if (POLY)
    line_far2<INF, true>(P.dr2, ADZ, (float)n_cut, SR, SZ);
  else
    base2<INF>(P.dr2, ADZ, S, SR, SZ);
  const u64 LA = add2(ADZ, dup(S.A));
  const u64 IL = rsq2(fma2(LA, LA, P.dr2));
  const u64 E = mul2(IL, IL), E2 = mul2(E, E);
  const u64 ER = mul2(E2, E), EZ = mul2(E2, IL);
  M.a0 = fma2(ER, dup(S.mu0), SR);
  M.b0 = mul2(ER, dup(S.sc0));
  M.a1 = fma2(EZ, dup(S.mu1), SZ);
  M.b1 = mul2(EZ, dup(S.sc1));
}

// The sums from the model's outputs.
template <int MODEL, bool RAW>
__device__ __forceinline__ void model_finish2(const Sep2& P, u64 ADZ, int n_cut, const Model2& M, u64 Y0, u64 Y1,
                                              u64& SR, u64& SZ) {
  SR = fma2(M.b0, Y0, M.a0);
  SZ = fma2(M.b1, Y1, M.a1);
  fix_dz0<MODEL == kModelWide4 && !RAW>(ADZ, P.dr2, (float)n_cut, SR, SZ);
  SZ = mulsign2(SZ, P.dz);
}

// Learned tail: one network call for the warp's 64 pairs (mlp_warp's two values of
// j are here the thread's two i).
template <int MODEL, bool FAR>
struct SurrForm {
  int n_cut;
  SurrW W;
  uint32_t* ibuf;
  const SurrConst& S;
  __device__ __forceinline__ void operator()(const Sep2& P, u64& SR, u64& SZ) const {
    const u64 ADZ = abs2(P.dz);
    Model2 M;
    model_stage2<MODEL, false, FAR>(P, ADZ, n_cut, S, M);
    float u[2][3], y[2][2];
#pragma unroll
    for (int c = 0; c < 3; ++c) upk(M.u[c], u[0][c], u[1][c]);
    mlp_warp<2>(W, ibuf, u, y);
    model_finish2<MODEL, false>(P, ADZ, n_cut, M, pk(y[0][0], y[1][0]), pk(y[0][1], y[1][1]), SR, SZ);
  }
};

// Correction-table tail (tail_table.cuh); READ: the table read (the exact reads
// belong to the nearest-image table, n0 = 0, stored raw).
template <int MODEL, int READ, bool FAR>
struct TableForm {
  static constexpr bool RAW = READ >= kReadCicExact;
  static_assert(!(RAW && model_poly(MODEL)), "the raw tables have no base");
  int n_cut;
  const SurrConst& S;
  const TableTail& Tab;
  __device__ __forceinline__ void operator()(const Sep2& P, u64& SR, u64& SZ) const {
    const u64 ADZ = abs2(P.dz);
    Model2 M;
    model_stage2<MODEL, RAW, FAR>(P, ADZ, n_cut, S, M);
    float u0, v0, u1, v1;
    upk(M.u[0], u0, v0);
    upk(M.u[1], u1, v1);
    const float2 r = table_read<READ>(Tab, u0, u1), s = table_read<READ>(Tab, v0, v1);
    model_finish2<MODEL, RAW>(P, ADZ, n_cut, M, pk(r.x, s.x), pk(r.y, s.y), SR, SZ);
  }
};

// ---- the stream-K driver over the upper triangle -----------------------------
// The tile width is kBJ / tpb: whole blocks (tpb = 1), or quarters (tpb = 4) when
// there are too few blocks to fill the GPU. A quarter's 32 steps are split once more, over sp units of
// 32 / sp steps (whole Kahan groups), when even the quarters leave CTAs' places empty.

// Quarter tiles are taken below this many 128 x 128 units per SM.
#ifndef STEPS_SYM_SPLIT
#define STEPS_SYM_SPLIT 64
#endif
// The most units that a quarter tile's steps are split over: it holds four Kahan groups.
#ifndef STEPS_SYM_MAX_STEP_SPLIT
#define STEPS_SYM_MAX_STEP_SPLIT 4
#endif
static_assert(STEPS_SYM_MAX_STEP_SPLIT >= 1 && 32 % STEPS_SYM_MAX_STEP_SPLIT == 0 &&
                  (32 / STEPS_SYM_MAX_STEP_SPLIT) % STEPS_KAHAN_GROUP == 0,
              "a unit's steps are whole Kahan groups");
inline void sym_split(int NB, int sms, bool steps, int& tpb, int& sp) {
  const long long blocks = (long long)NB * (NB + 1) / 2;
  tpb = blocks < STEPS_SYM_SPLIT * (long long)sms ? 4 : 1;
  sp = 1;
  while (steps && tpb == 4 && sp < STEPS_SYM_MAX_STEP_SPLIT &&
         blocks * tpb * sp * 2 <= (long long)sms * STEPS_SYM_MIN_BLOCKS)
    sp *= 2;
}

template <bool COMP>
struct SymShared {
  JTile2 T;
  float J[kSymThreads / 32 * (COMP ? 2 : 1) * kJRow];
};

template <bool KAHAN, bool TWO = false, bool COMP = false, class Form>
__device__ __forceinline__ void sym_stream_k(const float4* __restrict__ jA, const float4* __restrict__ jB, int n,
                                             int NB, int tpb, int sp, long long Ua, long long U, int C, SymShared<COMP>& sh,
                                             const FixAcc& F, const Form& form) {
  // the units [Ua, Ua + U) (all of them, or a rank's share), split over C CTAs
  const int c = blockIdx.x;
  const long long u0 = Ua + (long long)c * U / C;
  const long long u1 = Ua + (long long)(c + 1) * U / C;
  const int jt = kBJ / tpb, upb = tpb * sp, ks = jt / sp;  // units per block, steps per unit
  constexpr int kRow = (COMP ? 2 : 1) * kJRow;
  float* row = sh.J + (threadIdx.x >> 5) * kRow;
  long long u = u0;
  while (u < u1) {
    const int b = (int)checked_index(tri_row(u / upb, NB), NB);
    const int v0 = (int)checked_index(b * upb + (u - upb * tri_off(b, NB)), (long long)NB * upb);
    const int v1 = (int)min((long long)NB * upb, (long long)v0 + (u1 - u));
    const int i0 = row_i0(b), i1 = i0 + 32;
    const I2 I = load_i2(jA, jB, i0, i1, n);
    u64 sx = 0, sy = 0, sz = 0, cx = 0, cy = 0, cz = 0;
    for (int v = v0; v < v1; ++v) {
      const int t = v / sp, kb = (v - t * sp) * ks;
      __syncthreads();
      load_tile2<kSymThreads>(jA, jB, n, t, jt, sh.T);
      __syncthreads();
      const bool sym = t / tpb != b;
      JRing<COMP> ring;
      constexpr int kGroup = COMP ? kCompGroup : STEPS_KAHAN_GROUP;  // a power of two that divides a unit's steps
#pragma unroll 1
      for (int k0 = kb; k0 < kb + ks; k0 += STEPS_KAHAN_GROUP) {
        u64 gx = 0, gy = 0, gz = 0;
#pragma unroll 1
        for (int k = k0; k < k0 + STEPS_KAHAN_GROUP; ++k) {
          const int q = jslot(k);
          Sep2 P;
          separation2(I, sh.T, q, P);
          u64 SR, SZ;
          form(P, SR, SZ);
          const u64 m = sh.T.MH[q].x;
          const u64 MS = mul2(m, SR);
          gx = fma2(P.dx, MS, gx);
          gy = fma2(P.dy, MS, gy);
          gz = fma2(m, SZ, gz);
          if (sym) {
            const bool full = ((k + 1) & (kGroup - 1)) == 0;  // the group's last step: its sums stay where they are
            ring.take(P.dx, P.dy, I.m, mul2(I.m, SR), SZ, !full);
            if (COMP && full) ring.flush(row, k, k < kb + kGroup || (k & 31) < kGroup);
          }
        }
        if (!COMP && sym) ring.flush(row, k0 + STEPS_KAHAN_GROUP - 1, k0 == kb || (k0 & 31) == 0);
        acc2<KAHAN>(sx, cx, gx);
        acc2<KAHAN>(sy, cy, gy);
        acc2<KAHAN>(sz, cz, gz);
      }
      if (sym) {
        __syncthreads();  // every warp's row is written
        for (int s = threadIdx.x; s < jt; s += kSymThreads) {
          const int j = t * jt + s;
          if (j < n) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              FixValue f{0, 0};
#pragma unroll
              for (int w = 0; w < kSymThreads / 32; ++w) {
                f.sub(fix_value<TWO>(F, sh.J[w * kRow + 3 * s + q]));
                if (COMP) f.sub(fix_value<TWO>(F, sh.J[w * kRow + kJRow + 3 * s + q]));
              }
              fix_add<TWO>(F, q, j, f);
            }
          }
        }
      }
    }
    const u64 S[3] = {sx, sy, sz}, K[3] = {cx, cy, cz};
#pragma unroll
    for (int q = 0; q < 3; ++q) fix_add_rows<KAHAN, TWO>(F, q, i0, i1, S[q], K[q]);
    u += v1 - v0;
  }
}

// ---- kernels ---------------------------------------------------------------
template <bool KAHAN, bool LINE, bool FAR>
__global__ void __launch_bounds__(kSymThreads, FAR ? STEPS_SYM_FAR_MIN_BLOCKS : STEPS_SYM_MIN_BLOCKS)
pair_sym_kernel(const float4* __restrict__ jA, const float4* __restrict__ jB, int n, int n_cut, int NB, int tpb, int sp,
                long long Ua, long long U, int C, FixAcc F) {
  __shared__ SymShared<false> sh;
  sym_stream_k<KAHAN>(jA, jB, n, NB, tpb, sp, Ua, U, C, sh, F, PlainForm<LINE, FAR>{n_cut, (float)n_cut});
}

template <bool KAHAN, int MODEL, bool FAR>
__global__ void __launch_bounds__(kSymThreads, STEPS_SYM_SURR_MIN_BLOCKS)
pair_sym_surr_kernel(const float4* __restrict__ jA, const float4* __restrict__ jB, int n, int n_cut, int NB, int tpb, int sp,
                     long long Ua, long long U, int C, const SurrLane* __restrict__ wl, SurrConst S, FixAcc F) {
  __shared__ SymShared<false> sh;
  __shared__ __align__(16) uint32_t sWT[32 * kSurrStride];
  __shared__ __align__(16) uint32_t sIn[kSymThreads / 32][2 * kInWords];
  uint32_t* ibuf = sIn[threadIdx.x >> 5];
  mlp_zero_inputs<2>(ibuf);
  stage_surr_weights(wl, sWT);
  sym_stream_k<KAHAN>(jA, jB, n, NB, tpb, sp, Ua, U, C, sh, F,
                      SurrForm<MODEL, FAR>{n_cut, SurrW{sWT + (threadIdx.x & 31) * kSurrStride}, ibuf, S});
}

template <bool KAHAN, int MODEL, int READ, bool FAR>
__global__ void __launch_bounds__(kSymThreads, STEPS_SYM_TABLE_MIN_BLOCKS)
pair_sym_table_kernel(const float4* __restrict__ jA, const float4* __restrict__ jB, int n, int n_cut, int NB, int tpb, int sp,
                      long long Ua, long long U, int C, TableTail T, SurrConst S, FixAcc F) {
  __shared__ SymShared<false> sh;
  sym_stream_k<KAHAN>(jA, jB, n, NB, tpb, sp, Ua, U, C, sh, F, TableForm<MODEL, READ, FAR>{n_cut, S, T});
}

// ---- R^3 -------------------------------------------------------------------
// The R^3 pair force (eq. NewtonianForce, one image per pair) is symmetric as well. A
// pair costs about 26 FP32 operations and one rsqrt, so what is left around it counts:
// a lane takes four rows (two packed sets), so that the four 128-bit j loads, the
// ring's three shuffles and the loop serve four pairs, and one warp is a CTA. With two
// rows per lane the duplicated j words alone would keep the shared-memory pipe busier
// than the FP32 one. The row kernel (r3_pair.cuh) evaluates every ordered pair in 31 issue
// slots per 32 pairs: 3.39 ms per force at N = 65,536 against 2.97 here (2.85 with one-word sums and j-side
// groups of eight steps, which lost sums or digits that the row kernel kept).
#ifndef STEPS_SYM_R3_MIN_BLOCKS
#define STEPS_SYM_R3_MIN_BLOCKS 16  // resident CTAs (warps) per SM the kernel is compiled for
#endif
#ifndef STEPS_SYM_R3_UNROLL
#define STEPS_SYM_R3_UNROLL 4
#endif
constexpr int kSymR3Unroll = STEPS_SYM_R3_UNROLL;

template <bool KAHAN>
__global__ void __launch_bounds__(32, STEPS_SYM_R3_MIN_BLOCKS)
pair_sym_r3_kernel(const float4* __restrict__ jA, const float4* __restrict__ jB, int n, int NB, int tpb, long long U,
                   int C, FixAcc F) {
  constexpr int NS = kBI / 64;  // packed sets of two rows per lane
  __shared__ JTile2 T;
  __shared__ float row[2 * kJRow];
  const int c = blockIdx.x, lane = threadIdx.x;
  const long long u1 = (long long)(c + 1) * U / C;
  const int jt = kBJ / tpb;
  long long u = (long long)c * U / C;
  while (u < u1) {
    const int b = (int)checked_index(tri_row(u / tpb, NB), NB);
    const int t0 = (int)checked_index(b * tpb + (u - tpb * tri_off(b, NB)), (long long)NB * tpb);
    const int t1 = (int)min((long long)NB * tpb, (long long)t0 + (u1 - u));
    I2 I[NS];
    u64 S[NS][3], K[NS][3];
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int i0 = b * kBI + 64 * s + lane;
      I[s] = load_i2(jA, jB, i0, i0 + 32, n);
#pragma unroll
      for (int q = 0; q < 3; ++q) S[s][q] = K[s][q] = 0;
    }
    for (int t = t0; t < t1; ++t) {
      __syncwarp();
      load_tile2<32>(jA, jB, n, t, jt, T);
      __syncwarp();
      const bool sym = t / tpb != b;
      JRing<true> ring;
#pragma unroll 1
      for (int k0 = 0; k0 < jt; k0 += STEPS_KAHAN_GROUP) {
        u64 g[NS][3];
#pragma unroll
        for (int s = 0; s < NS; ++s) g[s][0] = g[s][1] = g[s][2] = 0;
#pragma unroll(kSymR3Unroll)
        for (int k = k0; k < k0 + STEPS_KAHAN_GROUP; ++k) {
          const int q = jslot(k);
          const ulonglong2 xy = T.XY[q], xyl = T.XYL[q], z = T.Z[q], mh = T.MH[q];
          u64 D[NS][3], R2[NS], RI[NS], HH[NS], Fr[NS];
          bool soft = false;
#pragma unroll
          for (int s = 0; s < NS; ++s) {
            D[s][0] = add2(sub2(I[s].xh, xy.x), sub2(I[s].xl, xyl.x));
            D[s][1] = add2(sub2(I[s].yh, xy.y), sub2(I[s].yl, xyl.y));
            D[s][2] = add2(sub2(I[s].zh, z.x), sub2(I[s].zl, z.y));
            R2[s] = fma2(D[s][0], D[s][0], fma2(D[s][1], D[s][1], mul2(D[s][2], D[s][2])));
            HH[s] = add2(I[s].h, mh.y);
            float ra, rb, ha, hb;
            upk(R2[s], ra, rb);
            upk(mul2(HH[s], HH[s]), ha, hb);
            soft = soft || ra < ha || rb < hb;
            RI[s] = rsq2(max2(R2[s], 1e-30f));
            Fr[s] = mul2(mul2(RI[s], RI[s]), RI[s]);
          }
          if (__any_sync(0xffffffffu, soft)) {
#pragma unroll
            for (int s = 0; s < NS; ++s) {
              const Soft2 h = soft2(HH[s]);
              Fr[s] = spline_value_r2(R2[s], RI[s], Fr[s], h.ih, h.nih, h.ih3);
            }
          }
#pragma unroll
          for (int s = 0; s < NS; ++s) {
            const u64 MF = mul2(mh.x, Fr[s]);
#pragma unroll
            for (int a = 0; a < 3; ++a) g[s][a] = fma2(D[s][a], MF, g[s][a]);
          }
          if (sym) {
            // the four pairs are added up first: the running sum takes one term per step
            u64 X[NS], V[3];
#pragma unroll
            for (int s = 0; s < NS; ++s) X[s] = mul2(I[s].m, Fr[s]);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
              V[a] = mul2(D[0][a], X[0]);
#pragma unroll
              for (int s = 1; s < NS; ++s) V[a] = fma2(D[s][a], X[s], V[a]);
            }
            ring.add(V);
            if ((k + 1) % kCompGroup == 0)
              ring.flush(row, k, (k & 31) < kCompGroup);
            else
              ring.shift();
          }
        }
#pragma unroll
        for (int s = 0; s < NS; ++s)
#pragma unroll
          for (int a = 0; a < 3; ++a) acc2<KAHAN>(S[s][a], K[s][a], g[s][a]);
      }
      if (sym) {
        __syncwarp();
        for (int s = lane; s < jt; s += 32) {
          const int j = t * jt + s;
          if (j < n) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              FixValue f{0, 0};
              f.sub(fix_value<true>(F, row[3 * s + q]));
              f.sub(fix_value<true>(F, row[kJRow + 3 * s + q]));
              fix_add<true>(F, q, j, f);
            }
          }
        }
      }
    }
#pragma unroll
    for (int s = 0; s < NS; ++s) {
      const int i0 = b * kBI + 64 * s + lane;
#pragma unroll
      for (int q = 0; q < 3; ++q) fix_add_rows<KAHAN, true>(F, q, i0, i0 + 32, S[s][q], K[s][q]);
    }
    u += t1 - t0;
  }
}

}  // namespace steps
