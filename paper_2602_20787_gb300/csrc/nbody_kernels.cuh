// O(N) kernels of the S1xR2 step (arXiv 2602.20787,
// eq. ComovingEquationsOfMotionCylindrical and the KDK leapfrog of Sect. 2.1).
#pragma once
#include <cstdint>

#include "pair_fp32.cuh"

namespace steps {
// The kernels below have internal linkage (static): every translation unit
// that includes this header gets its own copy.

constexpr int kErrNonFinite = 1;     // a force, position or momentum is not finite
constexpr int kErrBgRange = 2;       // a particle lies beyond the background table
constexpr int kErrZRange = 4;        // z left [0, L) by more than rounding
constexpr int kErrTreeRange = 8;     // a particle lies outside the octree's root cube
constexpr int kErrTreeStack = 16;    // an octree walk outgrew its stack

// The farthest from the axis, in units of L, that a finite window's packed words go: beyond dR of some
// 1e15 the products of a pair vanish in FP32, so nothing changes by it, but dR^2 stays finite, which the
// closed form of the image line relies on. (The infinite window's pair falls as 1 / dR^2 and the closed form is
// finite at any dR; R^3 has none: no cap.) Words that are not finite stay so.
constexpr float kPackCap = 6e18f;

// FP64 positions -> FP32 hi/lo words in units of L (see pair_fp32.cuh).
__device__ __forceinline__ void pack_one(double x, double y, double z, double m, double h, int i, double invL, float cap,
                                         float4* __restrict__ jA, float4* __restrict__ jB) {
  const double u[3] = {x * invL, y * invL, z * invL};
  float hi[3], lo[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    hi[c] = (float)u[c];
    lo[c] = (float)(u[c] - (double)hi[c]);
    if (c < 2 && fabsf(hi[c]) > cap && isfinite(hi[c])) {
      hi[c] = copysignf(cap, hi[c]);
      lo[c] = 0.0f;
    }
  }
  jA[i] = make_float4(hi[0], hi[1], hi[2], (float)m);
  jB[i] = make_float4(lo[0], lo[1], lo[2], (float)(h * invL));
}

static __global__ void pack_kernel(const double* __restrict__ x, const double* __restrict__ y,
                            const double* __restrict__ z, const double* __restrict__ m,
                            const double* __restrict__ h, int n, double invL, float cap, float4* __restrict__ jA,
                            float4* __restrict__ jB) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    pack_one(x[i], y[i], z[i], m[i], h[i], i, invL, cap, jA, jB);
}

// Background of eq. ComovingEquationsOfMotionCylindrical: returns F_h(rho) (< 0
// inside a homogeneous cylinder; the acceleration is -F_h along rho_hat).
// F_h = F_inf + dF, with F_inf the infinite cylinder (-2 pi G rho0 rho inside,
// -2 pi G rho0 R^2 / rho outside) and dF the smooth finite-height remainder,
// tabulated on a uniform grid (nodes -1 .. K+2) and read with 4-point Lagrange.
struct BgParams {
  int mode;            // STEPS_BG_* (3: the R^3 radial term +(4 pi G / 3) rho0 x)
  double two_pi_G_rho0;
  double R;
  const double* tab;   // dF at rho_k = k * dr, k = -1 .. K+2 (tab[0] is k = -1)
  int K;
  double inv_dr;
};

__device__ __forceinline__ double background_F(const BgParams& bg, double rho, int* err) {
  if (bg.mode == 0) return 0.0;
  double F = rho <= bg.R ? -bg.two_pi_G_rho0 * rho : -bg.two_pi_G_rho0 * bg.R * bg.R / rho;
  if (bg.mode == 1) {
    const double s = rho * bg.inv_dr;
    int k = (int)floor(s);
    if (k >= bg.K || !(s >= 0.0)) {
      atomicOr(err, kErrBgRange);
      k = bg.K - 1;
    }
    const double t = s - (double)k;  // in [0, 1)
    // Lagrange weights on nodes k-1, k, k+1, k+2 at offset t from node k
    const double wm = -t * (t - 1.0) * (t - 2.0) * (1.0 / 6.0);
    const double w0 = (t + 1.0) * (t - 1.0) * (t - 2.0) * 0.5;
    const double w1 = -(t + 1.0) * t * (t - 2.0) * 0.5;
    const double w2 = (t + 1.0) * t * (t - 1.0) * (1.0 / 6.0);
    const double* q = bg.tab + k;  // q[0] is node k-1
    F += wm * q[0] + w0 * q[1] + w1 * q[2] + w2 * q[3];
  }
  return F;
}

// The background term of particle (x, y, z) added to g (comoving field, a^3
// times the acceleration): the cylinder's F_h(rho) along -rho_hat (S1xR2), or
// the R^3 radial term +(4 pi G / 3) rho0 x = (2/3) (2 pi G rho0) x.
__device__ __forceinline__ void add_background(const BgParams& bg, double xi, double yi, double zi, double& g0,
                                               double& g1, double& g2, int* err) {
  if (bg.mode == 3) {
    const double c = bg.two_pi_G_rho0 * (2.0 / 3.0);
    g0 += c * xi;
    g1 += c * yi;
    g2 += c * zi;
    return;
  }
  const double rho = sqrt(xi * xi + yi * yi);
  if (rho > 0.0 && bg.mode != 0) {
    const double f = background_F(bg, rho, err) / rho;
    g0 -= f * xi;
    g1 -= f * yi;
  }
}

// Sum the stream-K partials of each i in CTA order (or read direct sums when
// NT == 0), scale to the comoving field
// g = a^3 (pair + background), store it, optionally kick p += g K and optionally
// write a = g / a^3 to an output.
// Radial correction of Sect. 2.4: g -= D(rho) rho_hat, D interpolated
// linearly between bin centres (k + 1/2) rmax / nb and held outside them.
// Radial correction of Sect. 2.4: g -= D(r) r_hat, D interpolated linearly
// between bin centres (k + 1/2) rmax / nb and held outside them; r is the
// cylindrical radius (S1xR2) or the distance from the origin (sph, R^3).
struct RadialCorr {
  const double* tab;  // nb bin means; null: no correction
  int nb;
  double rmax;
  int sph;
};

__device__ __forceinline__ void radial_correct(const RadialCorr& R, double x, double y, double z, double& g0,
                                               double& g1, double& g2) {
  if (!R.tab) return;
  const double rho = R.sph ? sqrt(x * x + y * y + z * z) : sqrt(x * x + y * y);
  if (!(rho > 0.0)) return;
  const double s = rho / R.rmax * R.nb - 0.5;
  double D;
  if (s <= 0.0) D = R.tab[0];
  else if (s >= R.nb - 1) D = R.tab[R.nb - 1];
  else {
    const int k = (int)s;
    const double t = s - k;
    D = (1.0 - t) * R.tab[k] + t * R.tab[k + 1];
  }
  g0 -= D * x / rho;
  g1 -= D * y / rho;
  if (R.sph) g2 -= D * z / rho;
}

// Accelerations a = g / a^3 written besides (x null: none), in the caller's order when perm maps
// the internal index to it.
struct AccelOut {
  double *x, *y, *z;
  double inv_a3;
  const int* perm;
};

// The common end of a finalize: the pair sums (sx, sy, sz) scaled to the
// comoving field g = a^3 (pair + background), the radial correction, the
// background; g stored, optionally p += g K, optionally a = g / a^3 written.
__device__ __forceinline__ void finish_particle(int i, double sx, double sy, double sz, double pair_scale,
                                                const BgParams& bg, const double* __restrict__ x,
                                                const double* __restrict__ y, const double* __restrict__ z,
                                                double* __restrict__ gx, double* __restrict__ gy,
                                                double* __restrict__ gz, double K, double* __restrict__ px,
                                                double* __restrict__ py, double* __restrict__ pz, const AccelOut& out,
                                                int* __restrict__ err, const RadialCorr& rc) {
  double g0 = pair_scale * sx, g1 = pair_scale * sy, g2 = pair_scale * sz;
  radial_correct(rc, x[i], y[i], z[i], g0, g1, g2);
  add_background(bg, x[i], y[i], z[i], g0, g1, g2, err);
  if (err && (!isfinite(g0) || !isfinite(g1) || !isfinite(g2))) atomicOr(err, kErrNonFinite);
  gx[i] = g0; gy[i] = g1; gz[i] = g2;
  if (px) {
    px[i] = fma(g0, K, px[i]);
    py[i] = fma(g1, K, py[i]);
    pz[i] = fma(g2, K, pz[i]);
  }
  if (out.x) {
    const int o = out.perm ? out.perm[i] : i;
    out.x[o] = g0 * out.inv_a3;
    out.y[o] = g1 * out.inv_a3;
    out.z[o] = g2 * out.inv_a3;
  }
}

// Threads per CTA of the O(N) kernels with FP64 work per particle (this finalize, its
// fixed-point form, the kick and drift). An SM's FP64 pipe takes a warp's instruction in 16 cycles, so what
// counts is how many SMs share the particles: at N = 2,048, CTAs of 256 leave 144 of 152 SMs
// idle (finalize 10.2 us, kick and drift 6.0).
inline int particle_threads(int n) { return n <= 152 * 8 * 32 ? 32 : 128; }

// The stream-K partials of evaluated row q, in CTA order.
__device__ __forceinline__ void row_sums(const double* __restrict__ part, int q, int NT, long long U, int C, double& sx,
                                         double& sy, double& sz) {
  const int b = q / kBI, l = q % kBI;
  const long long p_lo = (long long)b * NT, p_hi = p_lo + NT - 1;
  const int c_lo = cta_of_unit(p_lo, U, C), c_hi = cta_of_unit(p_hi, U, C);
  for (int c = c_lo; c <= c_hi; ++c) {
    const double* v = part + ((long long)b + c) * 3 * kBI;
    sx += v[l];
    sy += v[kBI + l];
    sz += v[2 * kBI + l];
  }
}

static __global__ void finalize_kernel(const double* __restrict__ part, int n, int NT, long long U, int C,
                                double pair_scale, BgParams bg, const double* __restrict__ x,
                                const double* __restrict__ y, const double* __restrict__ z, double* __restrict__ gx,
                                double* __restrict__ gy, double* __restrict__ gz, double K,
                                double* __restrict__ px, double* __restrict__ py, double* __restrict__ pz,
                                AccelOut out, int* __restrict__ err,
                                RadialCorr rc = RadialCorr{nullptr, 0, 0.0, 0}, int i0 = 0) {
  // rows [i0, n), i0 a multiple of kBI (all rows unless they are sharded); the
  // partials and direct sums are indexed from i0
  const int i = i0 + blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double sx = 0.0, sy = 0.0, sz = 0.0;
  if (NT == 0) {
    // direct sums (FP64 pair kernel, octree): C sets [3][n - i0]
    const long long q = i - i0, m = n - i0;
    for (int c = 0; c < C; ++c) {
      const double* v = part + 3 * m * c;
      sx += v[q];
      sy += v[m + q];
      sz += v[2 * m + q];
    }
  } else {
    row_sums(part, i - i0, NT, U, C, sx, sy, sz);
  }
  finish_particle(i, sx, sy, sz, pair_scale, bg, x, y, z, gx, gy, gz, K, px, py, pz, out, err, rc);
}

// First half of a KDK step for particle i with the field g: p += g K1, x += p D, z wrapped into
// [0, L) (wrap: S1xR2), the packed words. Products and sums are fused explicitly, so that a step's
// bits do not depend on the kernel that takes it.
struct DriftStep {
  double K1, D, L, invL;
  float cap;  // of the packed words
  int wrap;
};
__device__ __forceinline__ void kick_drift_one(int i, double g0, double g1, double g2, const DriftStep& S, double* x,
                                               double* y, double* z, double* px, double* py, double* pz,
                                               const double* __restrict__ m, const double* __restrict__ h,
                                               float4* __restrict__ jA, float4* __restrict__ jB, int* err) {
  const double qx = fma(g0, S.K1, px[i]), qy = fma(g1, S.K1, py[i]), qz = fma(g2, S.K1, pz[i]);
  px[i] = qx; py[i] = qy; pz[i] = qz;
  const double nx = fma(qx, S.D, x[i]), ny = fma(qy, S.D, y[i]);
  double nz = fma(qz, S.D, z[i]);
  if (S.wrap) {
    nz = fma(-S.L, floor(nz * S.invL), nz);
    if (nz >= S.L) nz -= S.L;
    if (nz < 0.0) nz = 0.0;
  }
  if (!isfinite(nx) || !isfinite(ny) || !isfinite(nz)) atomicOr(err, kErrNonFinite);
  x[i] = nx; y[i] = ny; z[i] = nz;
  pack_one(nx, ny, nz, m[i], h[i], i, S.invL, S.cap, jA, jB);
}

// A fixed-point sum as a double: hi in units of inv_scale, *lo (null: none) in units of 2^-40 of it.
__device__ __forceinline__ double fix_sum(unsigned long long hi, const unsigned long long* lo, double inv_scale) {
  const double s = (double)(long long)hi * inv_scale;
  return lo ? fma((double)(long long)*lo, inv_scale * 0x1p-40, s) : s;
}

// The end of a step and the beginning of the next in one pass: the finalize from the fixed-point
// sums [3][n] (lo: their low words or null), the kick K of the step that ends, then the kick and drift of the next, with the sums
// cleared for its force evaluation: one launch for two (7.8 and 5.1 us of 42 at N = 2,048).
static __global__ void finalize_fix_drift_kernel(unsigned long long* __restrict__ acc,
                                                 unsigned long long* __restrict__ lo, int n, double inv_scale,
                                                 double pair_scale, BgParams bg, double* __restrict__ x,
                                                 double* __restrict__ y, double* __restrict__ z,
                                                 double* __restrict__ gx, double* __restrict__ gy,
                                                 double* __restrict__ gz, double K, double* __restrict__ px,
                                                 double* __restrict__ py, double* __restrict__ pz,
                                                 const double* __restrict__ m, const double* __restrict__ h,
                                                 DriftStep S, float4* __restrict__ jA, float4* __restrict__ jB,
                                                 int* __restrict__ err) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double s[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const size_t o = (size_t)c * n + i;
    s[c] = fix_sum(acc[o], lo ? lo + o : nullptr, inv_scale);
    acc[o] = 0;
    if (lo) lo[o] = 0;
  }
  finish_particle(i, s[0], s[1], s[2], pair_scale, bg, x, y, z, gx, gy, gz, K, px, py, pz, AccelOut{}, err,
                  RadialCorr{nullptr, 0, 0.0, 0});
  kick_drift_one(i, gx[i], gy[i], gz[i], S, x, y, z, px, py, pz, m, h, jA, jB, err);
}

// Finalize from the fixed-point accumulators of the symmetric pair kernels
// (pair_sym.cuh), in units of 1 / scale, for the rows [i0, n): acc[3][stride]
// indexed from i0 (stride = n, i0 = 0 for every row; a rank's own rows of a
// sharded step have i0 = its first row and stride = its exchange chunk).
static __global__ void finalize_fix_kernel(const unsigned long long* __restrict__ acc,
                                           const unsigned long long* __restrict__ lo, int n, int i0, int stride,
                                           double inv_scale, double pair_scale, BgParams bg,
                                           const double* __restrict__ x, const double* __restrict__ y,
                                           const double* __restrict__ z, double* __restrict__ gx,
                                           double* __restrict__ gy, double* __restrict__ gz, double K,
                                           double* __restrict__ px, double* __restrict__ py,
                                           double* __restrict__ pz, AccelOut out, int* __restrict__ err) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = i0 + q;
  if (i >= n) return;
  const long long p = (long long)stride + q, r = 2 * (long long)stride + q;
  const double sx = fix_sum(acc[q], lo ? lo + q : nullptr, inv_scale);
  const double sy = fix_sum(acc[p], lo ? lo + p : nullptr, inv_scale);
  const double sz = fix_sum(acc[r], lo ? lo + r : nullptr, inv_scale);
  finish_particle(i, sx, sy, sz, pair_scale, bg, x, y, z, gx, gy, gz, K, px, py, pz, out, err,
                  RadialCorr{nullptr, 0, 0.0, 0});
}

// First half of a KDK step: p += g K1; x += p D; z wrapped into [0, L); repack. facc (may be
// null): the fixed-point sums [3][n] of the force evaluation that follows, set to zero (and lo,
// their low words).
static __global__ void kick_drift_pack_kernel(double* __restrict__ x, double* __restrict__ y,
                                       double* __restrict__ z, double* __restrict__ px,
                                       double* __restrict__ py, double* __restrict__ pz,
                                       const double* __restrict__ gx, const double* __restrict__ gy,
                                       const double* __restrict__ gz, const double* __restrict__ m,
                                       const double* __restrict__ h, int n, DriftStep S, float4* __restrict__ jA,
                                       float4* __restrict__ jB, int* __restrict__ err,
                                       unsigned long long* __restrict__ facc,
                                       unsigned long long* __restrict__ lo) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    if (facc) {
      facc[i] = 0;
      facc[(size_t)n + i] = 0;
      facc[2 * (size_t)n + i] = 0;
      if (lo) lo[i] = lo[(size_t)n + i] = lo[2 * (size_t)n + i] = 0;
    }
    kick_drift_one(i, gx[i], gy[i], gz[i], S, x, y, z, px, py, pz, m, h, jA, jB, err);
  }
}

// Deterministic reductions for the diagnostics: each block writes its partial
// sums of (m px, m py, m pz, m (x py - y px), m |p|^2 / 2, m) into part[block][6].
constexpr int kRedThreads = 256;
constexpr int kRedBlocks = 256;

static __global__ void diag_partial_kernel(const double* __restrict__ x, const double* __restrict__ y,
                                    const double* __restrict__ px, const double* __restrict__ py,
                                    const double* __restrict__ pz, const double* __restrict__ m, int n,
                                    double* __restrict__ part) {
  double v[6] = {0, 0, 0, 0, 0, 0};
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double mi = m[i];
    v[0] += mi * px[i];
    v[1] += mi * py[i];
    v[2] += mi * pz[i];
    v[3] += mi * (x[i] * py[i] - y[i] * px[i]);
    v[4] += 0.5 * mi * (px[i] * px[i] + py[i] * py[i] + pz[i] * pz[i]);
    v[5] += mi;
  }
  __shared__ double sh[kRedThreads / 32][6];
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    double s = v[q];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5][q] = s;
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    double s = 0.0;
    for (int w = 0; w < kRedThreads / 32; ++w) s += sh[w][threadIdx.x];
    part[blockIdx.x * 6 + threadIdx.x] = s;
  }
}

static __global__ void diag_final_kernel(const double* __restrict__ part, int nblocks, double* __restrict__ out) {
  if (threadIdx.x < 6) {
    double s = 0.0;
    for (int b = 0; b < nblocks; ++b) s += part[b * 6 + threadIdx.x];
    out[threadIdx.x] = s;
  }
}

// out[3][ni] = sum over chunks c (in order) of part[c][3][ni]
static __global__ void chunk_sum_kernel(const double* __restrict__ part, int ni, int chunks, double* __restrict__ out) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= ni) return;
  double s0 = 0.0, s1 = 0.0, s2 = 0.0;
  for (int c = 0; c < chunks; ++c) {
    const double* p = part + (long long)c * 3 * ni;
    s0 += p[q];
    s1 += p[ni + q];
    s2 += p[2 * (long long)ni + q];
  }
  out[q] = s0;
  out[ni + q] = s1;
  out[2 * (long long)ni + q] = s2;
}

// out3 (SoA, ni each) = pair_scale * pair + background at the listed i, / a^3
static __global__ void subset_finalize_kernel(const double* __restrict__ pairsum, int ni, const int64_t* __restrict__ idx,
                                       double pair_scale, BgParams bg, const double* __restrict__ x,
                                       const double* __restrict__ y, const double* __restrict__ z, double inv_a3,
                                       double* __restrict__ ox, double* __restrict__ oy, double* __restrict__ oz,
                                       int* __restrict__ err) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= ni) return;
  const int i = idx ? (int)idx[q] : q;
  double g0 = pair_scale * pairsum[q], g1 = pair_scale * pairsum[ni + q], g2 = pair_scale * pairsum[2 * ni + q];
  add_background(bg, x[i], y[i], z[i], g0, g1, g2, err);
  if (!isfinite(g0) || !isfinite(g1) || !isfinite(g2)) atomicOr(err, kErrNonFinite);
  ox[q] = g0 * inv_a3;
  oy[q] = g1 * inv_a3;
  oz[q] = g2 * inv_a3;
}

// ---------------------------------------------------------------------------
// Row sharding (Sect. 2.4's distributed direct engine, one rank per GPU). Each
// rank owns a contiguous range of internal rows; the only exchange of a step is
// the packed positions of every rank's rows, gathered between the drift and the
// force evaluation.
// The owned packed rows [k0, k0 + rows) -> send[chunk][2] = (jA, jB) per row,
// zero rows past the share, so every rank sends chunk rows.
static __global__ void shard_send_kernel(const float4* __restrict__ jA, const float4* __restrict__ jB, int k0,
                                         int rows, int chunk, float4* __restrict__ send) {
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < chunk; q += gridDim.x * blockDim.x) {
    const bool own = q < rows;
    send[2 * q] = own ? jA[k0 + q] : make_float4(0.f, 0.f, 0.f, 0.f);
    send[2 * q + 1] = own ? jB[k0 + q] : make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// The gathered recv[world][chunk][2] -> the packed arrays: rank r's rows are
// [off[r], off[r + 1]) (blockIdx.y = r).
static __global__ void shard_recv_kernel(const float4* __restrict__ recv, const int* __restrict__ off, int chunk,
                                         float4* __restrict__ jA, float4* __restrict__ jB) {
  const int r = blockIdx.y;
  const int o = off[r], rows = off[r + 1] - o;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < rows; q += gridDim.x * blockDim.x) {
    const long long src = 2 * ((long long)r * chunk + q);
    jA[o + q] = recv[src];
    jB[o + q] = recv[src + 1];
  }
}

}  // namespace steps
