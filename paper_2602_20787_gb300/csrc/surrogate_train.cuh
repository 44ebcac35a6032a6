// Training side of the learned far-image surrogate (this project's method; the
// paper sums the image tail directly, eq. ForceCylindrical).
//
// The tail of a pair is the part of the image window of eq. ForceCylindrical
// beyond the near images |k| <= n0 (wrapped frame, lengths in units of L). The
// surrogate writes it as
//   tail = B1 + E * (MLP(u) * sc + mu)            (z component times sign(dz))
// with B1 the continuum integral of the image cells plus the first
// Euler-Maclaurin end correction, E an envelope (e^3 for SR, e^(5/2) for SZ,
// e = 1 / (dR^2 + (n0 + 1/2 + |dz|)^2)), and a 3 -> 32 -> 32 -> 2 ReLU MLP of
// u = (2 min(dR, dR_max)/dR_max - 1, 4|dz| - 1, 2 min(h, n0+1/2)/(n0+1/2) - 1).
//
// Kernels here: exact FP64 tail sums (training targets), the FP64 base and
// envelope, and FP32 forward/backward/Adam. Gradients are accumulated per block
// and reduced in block order, so training is deterministic.
#pragma once
#include <cstdint>

#include "pair_fp32.cuh"

namespace steps {

constexpr int kH = 32;                                   // hidden width
constexpr int kNW = kH * 3 + kH + kH * kH + kH + 2 * kH + 2;  // 1250 weights
// offsets in the flat weight vector: W1[32][3], b1[32], W2[32][32], b2[32], W3[2][32], b3[2]
constexpr int kOW1 = 0, kOB1 = kOW1 + kH * 3, kOW2 = kOB1 + kH, kOB2 = kOW2 + kH * kH, kOW3 = kOB2 + kH,
              kOB3 = kOW3 + 2 * kH;

// Spline F(r,h)/r of eq. Force_spline_kernel in FP64 (support radius h).
__device__ __forceinline__ double spline_over_r_d(double r, double h) {
  if (r >= h) return 1.0 / (r * r * r);
  const double u = r / h, ih3 = 1.0 / (h * h * h);
  if (u < 0.5) return (32.0 / 3.0 + u * u * (32.0 * u - 38.4)) * ih3;
  const double u3 = u * u * u;
  return (64.0 / 3.0 - 48.0 * u + 38.4 * u * u - (32.0 / 3.0) * u3 - 1.0 / (15.0 * u3)) * ih3;
}

// The infinite window (Ncut -> infinity): images |k| <= kKInf are summed one by
// one, those beyond on each side by the continuum cells from kKInf + 1/2 with
// the near end's Euler-Maclaurin term (Newtonian there, as h << kKInf), which
// leaves an error of O(kKInf^-6).
constexpr int kKInf = 512;

// Both line ends beyond |k| = kKInf, added to (sr, sz), offsets o = dz + k.
__host__ __device__ __forceinline__ void line_ends_fp64(double R2, double dz, double& sr, double& sz) {
  const double top = kKInf + 0.5 + dz, bot = kKInf + 0.5 - dz;
  const double rt = sqrt(R2 + top * top), rb = sqrt(R2 + bot * bot), it = 1.0 / rt, ib = 1.0 / rb;
  const double it5 = it * it * it * it * it, ib5 = ib * ib * ib * ib * ib;
  sr += 1.0 / (rt * (rt + top)) - 3.0 * top * it5 / 24.0 + 1.0 / (rb * (rb + bot)) - 3.0 * bot * ib5 / 24.0;
  sz += it + (it * it * it - 3.0 * top * top * it5) / 24.0 - (ib + (ib * ib * ib - 3.0 * bot * bot * ib5) / 24.0);
}

// Exact tail sums of the window (|dz + k| < Ncut, |k| > n0) in FP64, units of L;
// n_cut = 0 is the infinite window.
// samples: ns x 3 (dR, dz, h); out: ns x 2 (SR, SZ).
static __global__ void tail_sums_fp64_kernel(const double* __restrict__ smp, int64_t ns, int n_cut, int n0,
                                             double* __restrict__ out) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < ns; s += (int64_t)gridDim.x * blockDim.x) {
    const double dR = smp[3 * s], dz = smp[3 * s + 1], h = smp[3 * s + 2];
    const double R2 = dR * dR;
    double sr = 0.0, sz = 0.0;
    if (n_cut == 0) {
      for (int k = n0 + 1; k <= kKInf; ++k) {
        const double op = dz + (double)k, om = dz - (double)k;
        const double fp = spline_over_r_d(sqrt(R2 + op * op), h), fm = spline_over_r_d(sqrt(R2 + om * om), h);
        sr += fp + fm;
        sz += op * fp + om * fm;
      }
      line_ends_fp64(R2, dz, sr, sz);
      out[2 * s] = sr;
      out[2 * s + 1] = sz;
      continue;
    }
    // walk outward from the near region on both sides
    for (int k = n0 + 1; k <= n_cut + 1; ++k) {
      const double op = dz + (double)k, om = dz - (double)k;
      if (fabs(op) < (double)n_cut) {
        const double f = spline_over_r_d(sqrt(R2 + op * op), h);
        sr += f;
        sz += op * f;
      }
      if (fabs(om) < (double)n_cut) {
        const double f = spline_over_r_d(sqrt(R2 + om * om), h);
        sr += f;
        sz += om * f;
      }
    }
    out[2 * s] = sr;
    out[2 * s + 1] = sz;
  }
}

// Continuum base B1 of one side: cells [lo, hi] of the unit-spaced images,
// f = (R^2 + z^2)^(-3/2) for SR and z f for SZ.
__host__ __device__ __forceinline__ void side_base_fp64(double R2, double lo, double hi, double& sr, double& sz) {
  const double rl = sqrt(R2 + lo * lo), rh = sqrt(R2 + hi * hi);
  const double il = 1.0 / rl, ih = 1.0 / rh;
  // Int f = (hi^2 - lo^2) / (rl rh (hi rl + lo rh)) (no cancellation at small R)
  const double IR = (hi - lo) * (hi + lo) / (rl * rh * (hi * rl + lo * rh));
  const double IZ = il - ih;
  const double il2 = il * il, ih2 = ih * ih, il5 = il2 * il2 * il, ih5 = ih2 * ih2 * ih;
  const double dRl = -3.0 * lo * il5, dRh = -3.0 * hi * ih5;
  const double dZl = il2 * il - 3.0 * lo * lo * il5, dZh = ih2 * ih - 3.0 * hi * hi * ih5;
  sr = IR - (dRh - dRl) / 24.0;
  sz = IZ - (dZh - dZl) / 24.0;
}

// B1 and the envelope for |dz| = adz (z component for positive dz).
__host__ __device__ __forceinline__ void tail_base_fp64(double dR, double adz, int n_cut, int n0, double& BR,
                                                        double& BZ, double& ER, double& EZ) {
  const double R2 = dR * dR, A = n0 + 0.5;
  const int kpos = n_cut - 1, kneg = adz > 0.0 ? n_cut : n_cut - 1;
  double r1, z1, r2, z2;
  side_base_fp64(R2, A + adz, kpos + 0.5 + adz, r1, z1);
  side_base_fp64(R2, A - adz, kneg + 0.5 - adz, r2, z2);
  BR = r1 + r2;
  BZ = z1 - z2;
  const double e = 1.0 / (R2 + (A + adz) * (A + adz));
  ER = e * e * e;
  EZ = e * e * sqrt(e);
}

// The same base with both far ends at infinity (the Ncut -> infinity window):
// per side the integral over [A +- |dz|, inf) plus the near end's
// Euler-Maclaurin term, Int = 1/(r (r + lo)) and 1/r.
__host__ __device__ __forceinline__ void tail_base_inf_fp64(double dR, double adz, int n0, double& BR, double& BZ,
                                                            double& ER, double& EZ) {
  const double R2 = dR * dR, A = n0 + 0.5;
  double br[2], bz[2];
  const double lo[2] = {A + adz, A - adz};
  for (int q = 0; q < 2; ++q) {
    const double l = lo[q], r = sqrt(R2 + l * l), il = 1.0 / r, il2 = il * il, il5 = il2 * il2 * il;
    br[q] = 1.0 / (r * (r + l)) - 3.0 * l * il5 / 24.0;
    bz[q] = il + (il2 * il - 3.0 * l * l * il5) / 24.0;
  }
  BR = br[0] + br[1];
  BZ = bz[0] - bz[1];
  const double e = 1.0 / (R2 + (A + adz) * (A + adz));
  ER = e * e * e;
  EZ = e * e * sqrt(e);
}

// Training samples: dR with density ~ dR (pairs in a plane), |dz| and h uniform, from the draws
// 3 s .. 3 s + 2 of the generator (SplitMix64 of state seed, a counter).
__device__ __forceinline__ double splitmix_uniform(uint64_t seed, uint64_t draw) {
  uint64_t z = seed + (draw + 1) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return (double)((z ^ (z >> 31)) >> 11) * (1.0 / 9007199254740992.0);
}
static __global__ void training_samples_kernel(uint64_t seed, int64_t ns, double dR_max, double A,
                                               double* __restrict__ smp) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < ns; s += (int64_t)gridDim.x * blockDim.x) {
    smp[3 * s] = dR_max * sqrt(splitmix_uniform(seed, 3 * s));
    smp[3 * s + 1] = 0.5 * splitmix_uniform(seed, 3 * s + 1);
    smp[3 * s + 2] = A * splitmix_uniform(seed, 3 * s + 2);
  }
}

// Training pairs: inputs u (FP32, ns x 3) and raw targets r = (tail - B1) / E
// (FP64, ns x 2, before the mean/scale normalisation) from exact tail sums
// (n_cut = 0: the infinite window over its base).
static __global__ void surrogate_dataset_kernel(const double* __restrict__ smp, const double* __restrict__ tail,
                                                int64_t ns, int n_cut, int n0, double dR_max,
                                                float* __restrict__ u, double* __restrict__ r) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < ns; s += (int64_t)gridDim.x * blockDim.x) {
    const double dR = smp[3 * s], adz = fabs(smp[3 * s + 1]), h = smp[3 * s + 2];
    double BR, BZ, ER, EZ;
    if (n_cut == 0)
      tail_base_inf_fp64(dR, adz, n0, BR, BZ, ER, EZ);
    else
      tail_base_fp64(dR, adz, n_cut, n0, BR, BZ, ER, EZ);
    const double A = n0 + 0.5;
    u[3 * s] = (float)(2.0 * fmin(dR, dR_max) / dR_max - 1.0);
    u[3 * s + 1] = (float)(4.0 * adz - 1.0);
    u[3 * s + 2] = (float)(2.0 * fmin(h, A) / A - 1.0);
    const double sg = smp[3 * s + 1] < 0.0 ? -1.0 : 1.0;
    r[2 * s] = (tail[2 * s] - BR) / ER;
    r[2 * s + 1] = (sg * tail[2 * s + 1] - BZ) / EZ;
  }
}

// Normalised FP32 targets t = (r - mu) / sc.
static __global__ void surrogate_normalise_kernel(const double* __restrict__ r, int64_t ns, double mu0, double mu1,
                                                  double sc0, double sc1, float* __restrict__ t) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < ns; s += (int64_t)gridDim.x * blockDim.x) {
    t[2 * s] = (float)((r[2 * s] - mu0) / sc0);
    t[2 * s + 1] = (float)((r[2 * s + 1] - mu1) / sc1);
  }
}

// ---------------------------------------------------------------------------
// FP32 MLP training. A block of kTrainCta threads takes kTrainThreads samples of the
// minibatch and writes their summed gradient to gpart[block][kNW].
//
// What bounds a step is latency: 4,096 samples are 64 blocks of a few thousand cycles, 1,200
// times in a row. Four threads share a sample (8 of 32 neurons each, two per packed
// FP32x2 operation), the weights lie in shared memory in both orders so that either
// direction reads the 8 it needs in two 128-bit broadcasts, and activations and deltas
// lie unit-major, so that the gradients read four samples per 128-bit load and a thread's
// tile of 2 x 2 weights shares them. With one thread per sample and the weights read
// through L1 the kernel took 19.8 us, the reduction, whose loads waited for each other, 6.4.
// Every sum keeps its order (inputs, samples, blocks ascending), so the trained weights
// keep their bits.
// ---------------------------------------------------------------------------
constexpr int kTrainThreads = 64;              // samples of a block
constexpr int kTrainCta = 4 * kTrainThreads;   // its threads
constexpr int kTrainRow = kTrainThreads + 4;   // row stride: 128-bit reads of 8 rows hit 32 banks
constexpr int kTrainT = kH + 4;                // row stride of the transposed W2

// v[0 .. 7] += x * w[0 .. 7] as four packed FMAs
__device__ __forceinline__ void axpy8(u64 (&v)[4], float x, const float* w) {
  const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(w), b = *reinterpret_cast<const ulonglong2*>(w + 4);
  const u64 X = pk(x, x);
  v[0] = fma2(a.x, X, v[0]);
  v[1] = fma2(a.y, X, v[1]);
  v[2] = fma2(b.x, X, v[2]);
  v[3] = fma2(b.y, X, v[3]);
}

// The sample of a thread (threads of the first half: target g, and inputs 2 g and, g = 0, 1).
struct TrainSample {
  bool valid;
  float tg, i0, i1;
};
__device__ __forceinline__ TrainSample load_sample(const float* __restrict__ u, const float* __restrict__ t,
                                                   const int* __restrict__ order, int64_t first, int64_t count,
                                                   int block) {
  const int s = threadIdx.x % kTrainThreads, g = threadIdx.x / kTrainThreads;
  const int64_t q = (int64_t)block * kTrainThreads + s;
  TrainSample in{q < count, 0.f, 0.f, 0.f};
  if (g < 2 && in.valid) {
    const int64_t k = order ? (int64_t)order[first + q] : first + q;
    in.tg = t[2 * k + g];
    in.i0 = u[3 * k + 2 * g];
    if (g == 0) in.i1 = u[3 * k + 1];
  }
  return in;
}

struct TrainShared {
  __align__(16) float sW[kNW + 2];
  __align__(16) float sT[kH * kTrainT];
  __align__(16) float s_in[3][kTrainRow], s_a1[kH][kTrainRow], s_d1[kH][kTrainRow], s_a2[kH][kTrainRow],
      s_d2[kH][kTrainRow], s_e[2][kTrainRow], s_loss[kTrainThreads];
};

// Summed gradient and loss of a block's samples. The weights are read past L1: inside
// mlp_epoch_kernel other SMs write them.
__device__ __forceinline__ void fwd_bwd_block(TrainShared& sh, const float* w, const TrainSample& in, int block,
                                              float* __restrict__ gpart, float* __restrict__ lpart) {
  static_assert(kH == 32 && kOW2 % 4 == 0, "eight neurons per thread, 128-bit reads of W2");
  const int tid = threadIdx.x, s = tid % kTrainThreads, g = tid / kTrainThreads, o0 = 8 * g;
  if (g < 2) {
    sh.s_in[2 * g][s] = in.i0;
    if (g == 0) sh.s_in[1][s] = in.i1;
  }
#pragma unroll
  for (int r = 0; r < (kNW + kTrainCta - 1) / kTrainCta; ++r) {
    const int p = r * kTrainCta + tid;
    if (p < kNW) {
      const float v = __ldcg(w + p);
      sh.sW[p] = v;
      if (p >= kOW2 && p < kOB2) sh.sT[((p - kOW2) % kH) * kTrainT + (p - kOW2) / kH] = v;
    }
  }
  __syncthreads();
  // forward; ReLU'(z) is read from a = relu(z) > 0 (the same mask)
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int o = o0 + j;
    float v = sh.sW[kOB1 + o];
#pragma unroll
    for (int k = 0; k < 3; ++k) v = fmaf(sh.sW[kOW1 + o * 3 + k], sh.s_in[k][s], v);
    sh.s_a1[o][s] = fmaxf(v, 0.f);
  }
  __syncthreads();
  float a2[8];
  {
    u64 v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = pk(sh.sW[kOB2 + o0 + 2 * j], sh.sW[kOB2 + o0 + 2 * j + 1]);
#pragma unroll 8
    for (int k = 0; k < kH; ++k) axpy8(v, sh.s_a1[k][s], sh.sT + k * kTrainT + o0);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      upk(v[j], a2[2 * j], a2[2 * j + 1]);
      a2[2 * j] = fmaxf(a2[2 * j], 0.f);
      a2[2 * j + 1] = fmaxf(a2[2 * j + 1], 0.f);
      sh.s_a2[o0 + 2 * j][s] = a2[2 * j];
      sh.s_a2[o0 + 2 * j + 1][s] = a2[2 * j + 1];
    }
  }
  __syncthreads();
  if (g < 2) {
    float v = sh.sW[kOB3 + g];
#pragma unroll
    for (int k = 0; k < kH; ++k) v = fmaf(sh.sW[kOW3 + g * kH + k], sh.s_a2[k][s], v);
    sh.s_e[g][s] = in.valid ? (v - in.tg) : 0.f;
  }
  __syncthreads();
  // backward: d2 = (W3^T e) * relu'(z2), d1 = (W2^T d2) * relu'(z1)
  const float e[2] = {sh.s_e[0][s], sh.s_e[1][s]};
  const float* W3 = sh.sW + kOW3;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int k = o0 + j;
    const float d = W3[k] * e[0] + W3[kH + k] * e[1];
    sh.s_d2[k][s] = a2[j] > 0.f ? d : 0.f;
  }
  if (g == 0) sh.s_loss[s] = 0.5f * (e[0] * e[0] + e[1] * e[1]);
  __syncthreads();
  {
    u64 v[4] = {0, 0, 0, 0};
#pragma unroll 8
    for (int o = 0; o < kH; ++o) axpy8(v, sh.s_d2[o][s], sh.sW + kOW2 + o * kH + o0);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float x, y;
      upk(v[j], x, y);
      sh.s_d1[o0 + 2 * j][s] = sh.s_a1[o0 + 2 * j][s] > 0.f ? x : 0.f;
      sh.s_d1[o0 + 2 * j + 1][s] = sh.s_a1[o0 + 2 * j + 1][s] > 0.f ? y : 0.f;
    }
  }
  __syncthreads();
  // block partial gradient, samples in order. W2: rows o, o + 16, columns k, k + 16
  float* gp = gpart + (int64_t)block * kNW;
  {
    const int k = tid % 16, o = tid / 16;
    float c00 = 0.f, c01 = 0.f, c10 = 0.f, c11 = 0.f;
#pragma unroll 4
    for (int r = 0; r < kTrainThreads; r += 4) {
      const float4 A0 = *reinterpret_cast<const float4*>(&sh.s_a1[k][r]), A1 = *reinterpret_cast<const float4*>(&sh.s_a1[k + 16][r]);
      const float4 D0 = *reinterpret_cast<const float4*>(&sh.s_d2[o][r]), D1 = *reinterpret_cast<const float4*>(&sh.s_d2[o + 16][r]);
      c00 = fmaf(D0.w, A0.w, fmaf(D0.z, A0.z, fmaf(D0.y, A0.y, fmaf(D0.x, A0.x, c00))));
      c01 = fmaf(D0.w, A1.w, fmaf(D0.z, A1.z, fmaf(D0.y, A1.y, fmaf(D0.x, A1.x, c01))));
      c10 = fmaf(D1.w, A0.w, fmaf(D1.z, A0.z, fmaf(D1.y, A0.y, fmaf(D1.x, A0.x, c10))));
      c11 = fmaf(D1.w, A1.w, fmaf(D1.z, A1.z, fmaf(D1.y, A1.y, fmaf(D1.x, A1.x, c11))));
    }
    float* d = gp + kOW2 + o * kH + k;
    d[0] = c00;
    d[16] = c01;
    d[16 * kH] = c10;
    d[16 * kH + 16] = c11;
  }
  // the other weights: sums over the samples of a row product (W1, W3) or of a row (b1, b2, b3)
  constexpr int kRest = kNW - kH * kH;
  static_assert(kRest <= kTrainCta - 1, "one of the other weights per thread, the last thread sums the loss");
  if (tid < kRest) {
    const int p = tid < kOW2 ? tid : tid + kH * kH;
    const float *A, *B = nullptr;
    if (p < kOB1) {
      A = sh.s_d1[p / 3];
      B = sh.s_in[p % 3];
    } else if (p < kOW2) {
      A = sh.s_d1[p - kOB1];
    } else if (p < kOW3) {
      A = sh.s_d2[p - kOB2];
    } else if (p < kOB3) {
      A = sh.s_e[(p - kOW3) / kH];
      B = sh.s_a2[(p - kOW3) % kH];
    } else {
      A = sh.s_e[p - kOB3];
    }
    float c = 0.f;
    if (B) {
#pragma unroll 4
      for (int r = 0; r < kTrainThreads; r += 4) {
        const float4 a = *reinterpret_cast<const float4*>(A + r), b = *reinterpret_cast<const float4*>(B + r);
        c = fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, c))));
      }
    } else {
#pragma unroll 4
      for (int r = 0; r < kTrainThreads; r += 4) {
        const float4 a = *reinterpret_cast<const float4*>(A + r);
        c = (((c + a.x) + a.y) + a.z) + a.w;
      }
    }
    gp[p] = c;
  } else if (tid == kTrainCta - 1) {
    float l = 0.f;
    for (int r = 0; r < kTrainThreads; ++r) l += sh.s_loss[r];
    lpart[block] = l;
  }
}

static __global__ void __launch_bounds__(kTrainCta)
mlp_fwd_bwd_kernel(const float* __restrict__ w, const float* __restrict__ u, const float* __restrict__ t,
                   const int* __restrict__ order, int64_t first, int64_t count, float* __restrict__ gpart,
                   float* __restrict__ lpart) {
  __shared__ TrainShared sh;
  fwd_bwd_block(sh, w, load_sample(u, t, order, first, count, blockIdx.x), blockIdx.x, gpart, lpart);
}

struct AdamCfg {
  float lr, beta1, beta2, eps;
};
__device__ __forceinline__ void adam_update(float g, const AdamCfg& A, float c1, float c2, float& w, float& m1,
                                            float& m2) {
  const float a = fmaf(1.f - A.beta1, g, A.beta1 * m1);
  const float v = fmaf((1.f - A.beta2) * g, g, A.beta2 * m2);
  m1 = a;
  m2 = v;
  w -= A.lr * (a / c1) / (sqrtf(v / c2) + A.eps);
}

// Sum the block partials of each weight in block order, divide by the batch,
// and (when adam) take an Adam step. grad_out (optional) receives the gradient.
// One warp per CTA: the 1,250 sums spread over 40 SMs, and 32 of a sum's loads are in flight.
constexpr int kAdamThreads = 32, kAdamLoads = 32;
static __global__ void __launch_bounds__(kAdamThreads)
mlp_reduce_adam_kernel(const float* __restrict__ gpart, int nblocks, float inv_batch, float* __restrict__ w,
                       float* __restrict__ m1, float* __restrict__ m2, AdamCfg A, float c1, float c2, int adam,
                       float* __restrict__ grad_out) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= kNW) return;
  float M1 = 0.f, M2 = 0.f, W = 0.f;
  if (adam) {
    M1 = m1[p];
    M2 = m2[p];
    W = w[p];
  }
  float g = 0.f;
  for (int b = 0; b < nblocks; b += kAdamLoads) {
    float v[kAdamLoads];
#pragma unroll
    for (int k = 0; k < kAdamLoads; ++k) v[k] = b + k < nblocks ? gpart[(int64_t)(b + k) * kNW + p] : 0.f;
#pragma unroll
    for (int k = 0; k < kAdamLoads; ++k)
      if (b + k < nblocks) g += v[k];
  }
  g *= inv_batch;
  if (grad_out) grad_out[p] = g;
  if (adam) {
    adam_update(g, A, c1, c2, W, M1, M2);
    m1[p] = M1;
    m2[p] = M2;
    w[p] = W;
  }
}

// ---------------------------------------------------------------------------
// All steps of an epoch in one cooperative launch, a block of samples per CTA: between the
// gradient of a step and its update, and between that and the next step, the CTAs meet at a
// barrier in memory, and a CTA's next samples are fetched meanwhile. As two launches per step
// (the kernels above) a step of 64 blocks took 14 us, most of it launch latency and cold loads.
// ---------------------------------------------------------------------------
constexpr unsigned kBarrierSpins = 1u << 22;  // polls (of some 0.5 us) before a barrier gives up

// Every CTA of the grid arrives (target: arrivals once all have). A wait that runs out sets *fail; the
// waits after it in the same epoch end after 1,024 polls, half a millisecond each (the flag is not
// looked at before: that would cost every barrier a round trip), and later epochs do nothing.
__device__ __forceinline__ void grid_barrier(unsigned* bar, unsigned target, int* fail) {
  __syncthreads();
  if (threadIdx.x == 0) {
    // release: the CTA's writes (ordered before by the block's barrier) are visible with the arrival
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    unsigned seen = 0;
    for (unsigned k = 0; k < kBarrierSpins; ++k) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
      if (seen >= target || ((k & 1023u) == 1023u && atomicAdd(fail, 0) != 0)) break;
    }
    if (seen < target) atomicExch(fail, 1);
  }
  __syncthreads();
}

constexpr int kRedRow = kTrainThreads + 1;  // row stride of the gradient tile (32 weights x 64 blocks)
static __global__ void __launch_bounds__(kTrainCta)
mlp_epoch_kernel(float* w, const float* __restrict__ u, const float* __restrict__ t, const int* __restrict__ order,
                 int64_t ntrain, int batch, float* gpart, float* lpart, float* m1, float* m2, AdamCfg A,
                 const float2* __restrict__ corr, unsigned* bar, int* fail) {
  __shared__ TrainShared sh;
  static_assert(sizeof(sh.s_a1) >= sizeof(float) * 32 * kRedRow, "the gradient tile takes the activations' place");
  float* red = &sh.s_a1[0][0];
  unsigned target = 0;
  int step = 0;
  if (*static_cast<volatile int*>(fail) != 0) return;  // a barrier of an earlier epoch ran out
  TrainSample in = load_sample(u, t, order, 0, min((int64_t)batch, ntrain), blockIdx.x);
  for (int64_t first = 0; first < ntrain; first += batch, ++step) {
    const int64_t count = min((int64_t)batch, ntrain - first), rest = ntrain - first - count;
    const int nblk = (int)((count + kTrainThreads - 1) / kTrainThreads);
    if ((int)blockIdx.x < nblk) fwd_bwd_block(sh, w, in, blockIdx.x, gpart, lpart);
    in = load_sample(u, t, order, first + count, min((int64_t)batch, rest), blockIdx.x);
    grid_barrier(bar, target += gridDim.x, fail);
    const int lane = threadIdx.x % 32, r0 = threadIdx.x / 32;
    for (int p0 = 32 * blockIdx.x; p0 < kNW; p0 += 32 * gridDim.x) {
      const int p = p0 + lane;
      float g = 0.f;
      for (int b0 = 0; b0 < nblk; b0 += kTrainThreads) {
        const int nb = min(kTrainThreads, nblk - b0);
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kTrainThreads; r += kTrainCta / 32) {
          const int b = r + r0;
          if (b < nb && p < kNW) red[lane * kRedRow + b] = __ldcg(gpart + (int64_t)(b0 + b) * kNW + p);
        }
        __syncthreads();
        if (r0 == 0 && p < kNW) {
#pragma unroll 16
          for (int b = 0; b < nb; ++b) g += red[lane * kRedRow + b];
        }
      }
      if (r0 == 0 && p < kNW) {
        const float2 c = corr[step];
        float W = __ldcg(w + p), M1 = m1[p], M2 = m2[p];
        adam_update(g * (1.0f / (float)count), A, c.x, c.y, W, M1, M2);
        m1[p] = M1;
        m2[p] = M2;
        w[p] = W;
      }
    }
    grid_barrier(bar, target += gridDim.x, fail);
  }
}

static __global__ void sum_floats_kernel(const float* __restrict__ x, int n, float scale, float* __restrict__ out) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    float s = 0.f;
    for (int i = 0; i < n; ++i) s += x[i];
    *out = s * scale;
  }
}

}  // namespace steps
