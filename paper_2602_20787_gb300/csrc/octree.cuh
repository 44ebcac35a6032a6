// Octree force (arXiv 2602.20787, Sect. 2.4 "Octree"): a Barnes-Hut tree of
// the S1xR2 volume, re-drawn in a random frame at every force evaluation.
//
// Frame. x' = c x - s y, y' = s x + c y (c, s = cos, sin phi), z' = z + zeta
// (minus L when >= L). The root is a cube of side S = 2 max(L, 2 R_sim) centred
// at (0, 0, L/2); normalised coordinates u = (x'/S + 1/2, y'/S + 1/2,
// (z' - L/2)/S + 1/2) lie in [0, 1) and are rounded to FP32. 21 bits per axis
// give a 63-bit Morton key (x bit b at key bit 3b + 2, y at 3b + 1, z at 3b).
//
// Build (all on the GPU). The keys are sorted by a stable LSD radix sort of
// eight 8-bit digits from caller order, so equal keys keep caller order. The
// tree is built level by level from the root: an active node's eight child
// ranges are found by binary search in the sorted keys, and one scan numbers
// the non-empty children (consecutively per parent) and the next level's
// active nodes (more than `leaf` particles, depth < 21). Moments are summed
// bottom-up in FP64, level by level: mass, centre of mass (x, y in the
// particles' frame, z in the tree frame and shifted back by zeta) and the
// largest softening. Each node is packed as a pseudo-particle in the layout of
// the pair kernels (hi/lo position over L, mass, h/L).
//
// Walk. One warp per group of 32 consecutive particles in key order (several at small
// N), all lanes on one shared stack, up to 32 nodes a step: a lane takes a node and tests it
// against the group's particles one by one. (All lanes on one node waited for the node's
// three dependent loads from L2, some 3,500 times per group: 9.58 ms at N = 262,144 against
// 8.94, 1.28 against 1.04 at 20,000.) A node is opened for the group when any particle opens
// it: s^2 >= theta^2 d^2, or |d| - (sqrt(3)/2) s <= hu_i + hu_max (d: offset of u
// from the node centre with z wrapped to the nearest image, hu = h / S). The
// test is evaluated in FP32 with exactly rounded operations in the order
// written, so it is reproducible off the GPU. An accepted node, or the
// particles of an opened leaf, are appended to the warp's interaction list in
// shared memory; full lists are evaluated by all 32 lanes with the pair form
// of the correction-table tail over the infinite window (near images
// |k| <= n0 exact, the rest from the table), exactly as the direct kernel
// evaluates a j-tile.
#pragma once
#include <algorithm>
#include <cstdint>

#include "pair_sym.cuh"
#include "tail_table.cuh"

namespace steps {

constexpr int kTreeDepth = 21;
constexpr int kSortThreads = 256;
constexpr int kSortRounds = 8;
constexpr int kSortTile = kSortThreads * kSortRounds;  // keys per sort tile
// Groups (warps) per CTA of the walk: one, as groups differ in work and a CTA holds its place until its
// slowest is done (four: 8.77 ms at N = 262,144 and 1.04 at 20,000, one: 7.90 and 0.94).
#ifndef STEPS_TREE_WARPS
#define STEPS_TREE_WARPS 1
#endif
#ifndef STEPS_TREE_LIST
#define STEPS_TREE_LIST 128   // interaction-list entries per warp (>= 64)
#endif
constexpr int kWalkWarps = STEPS_TREE_WARPS;
// Stack of a warp's walk. Going down one node at a time needs 7 * 21 + 1 entries (kWalkReserve);
// the rest lets the walk take up to 32 nodes a step (7 entries more each).
constexpr int kWalkStack = 512;
constexpr int kWalkReserve = 7 * kTreeDepth + 1;
static_assert((kWalkStack - kWalkReserve) / 7 >= 32, "the first steps take 32 nodes");
constexpr int kWalkList = STEPS_TREE_LIST;
static_assert(kWalkList >= 64, "a list must take 32 nodes or particles after a flush check");

struct TreeFrame {
  double c, s, zeta, L, halfL, invS;
};

struct TreeCrit {
  float Lu, hLu, th2;  // period and half period in root units (infinite for R^3), theta^2
};

// The R^3 frame (Sect. 2.4): the domain centre moved to cen, the frame rotated
// by the matrix R (row-major), root side S = 4 R_sim centred at cen.
struct TreeFrame3 {
  double cen[3], R[9], invS;
};

__device__ __forceinline__ uint64_t spread3(uint32_t v) {
  uint64_t x = v & 0x1fffffu;
  x = (x | (x << 32)) & 0x1f00000000ffffull;
  x = (x | (x << 16)) & 0x1f0000ff0000ffull;
  x = (x | (x << 8)) & 0x100f00f00f00f00full;
  x = (x | (x << 4)) & 0x10c30c30c30c30c3ull;
  x = (x | (x << 2)) & 0x1249249249249249ull;
  return x;
}

__device__ __forceinline__ uint32_t compact3(uint64_t x) {
  x &= 0x1249249249249249ull;
  x = (x | (x >> 2)) & 0x10c30c30c30c30c3ull;
  x = (x | (x >> 4)) & 0x100f00f00f00f00full;
  x = (x | (x >> 8)) & 0x1f0000ff0000ffull;
  x = (x | (x >> 16)) & 0x1f00000000ffffull;
  x = (x | (x >> 32)) & 0x1fffffull;
  return (uint32_t)x;
}

// Tree-frame coordinates of the particles (internal order): u4[i] = (u, hu);
// the key and the internal index go to caller position perm[i], the input
// order of the stable sort. zt[i] = z' in the tree frame.
static __global__ void tree_frame_kernel(const double* __restrict__ x, const double* __restrict__ y,
                                         const double* __restrict__ z, const double* __restrict__ h,
                                         const int* __restrict__ perm, int n, TreeFrame F, float4* __restrict__ u4,
                                         double* __restrict__ zt, uint64_t* __restrict__ key,
                                         int* __restrict__ val, int* __restrict__ err) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double xr = __fma_rn(F.c, x[i], -__dmul_rn(F.s, y[i]));
    const double yr = __fma_rn(F.s, x[i], __dmul_rn(F.c, y[i]));
    double zr = __dadd_rn(z[i], F.zeta);
    if (zr >= F.L) zr = __dsub_rn(zr, F.L);
    const float ux = __double2float_rn(__fma_rn(xr, F.invS, 0.5));
    const float uy = __double2float_rn(__fma_rn(yr, F.invS, 0.5));
    const float uz = __double2float_rn(__fma_rn(__dsub_rn(zr, F.halfL), F.invS, 0.5));
    const float hu = __double2float_rn(__dmul_rn(h[i], F.invS));
    const bool inside = ux >= 0.0f && ux < 1.0f && uy >= 0.0f && uy < 1.0f && uz >= 0.0f && uz < 1.0f;
    if (!inside) atomicOr(err, kErrTreeRange);
    const float cx = inside ? ux : 0.0f, cy = inside ? uy : 0.0f, cz = inside ? uz : 0.0f;
    const uint32_t qx = (uint32_t)__fmul_rn(cx, 2097152.0f), qy = (uint32_t)__fmul_rn(cy, 2097152.0f),
                   qz = (uint32_t)__fmul_rn(cz, 2097152.0f);
    u4[i] = make_float4(ux, uy, uz, hu);
    zt[i] = zr;
    const int c = perm[i];
    key[c] = (spread3(qx) << 2) | (spread3(qy) << 1) | spread3(qz);
    val[c] = i;
  }
}

// The same for the R^3 frame: u = R (x - cen) / S + 1/2, with the explicit
// fma/mul sequence; zt[i] = z[i] (no period).
static __global__ void tree_frame_r3_kernel(const double* __restrict__ x, const double* __restrict__ y,
                                            const double* __restrict__ z, const double* __restrict__ h,
                                            const int* __restrict__ perm, int n, TreeFrame3 F,
                                            float4* __restrict__ u4, double* __restrict__ zt,
                                            uint64_t* __restrict__ key, int* __restrict__ val, int* __restrict__ err) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double dx = __dsub_rn(x[i], F.cen[0]), dy = __dsub_rn(y[i], F.cen[1]), dz = __dsub_rn(z[i], F.cen[2]);
    const double xr = __fma_rn(F.R[0], dx, __fma_rn(F.R[1], dy, __dmul_rn(F.R[2], dz)));
    const double yr = __fma_rn(F.R[3], dx, __fma_rn(F.R[4], dy, __dmul_rn(F.R[5], dz)));
    const double zr = __fma_rn(F.R[6], dx, __fma_rn(F.R[7], dy, __dmul_rn(F.R[8], dz)));
    const float ux = __double2float_rn(__fma_rn(xr, F.invS, 0.5));
    const float uy = __double2float_rn(__fma_rn(yr, F.invS, 0.5));
    const float uz = __double2float_rn(__fma_rn(zr, F.invS, 0.5));
    const float hu = __double2float_rn(__dmul_rn(h[i], F.invS));
    const bool inside = ux >= 0.0f && ux < 1.0f && uy >= 0.0f && uy < 1.0f && uz >= 0.0f && uz < 1.0f;
    if (!inside) atomicOr(err, kErrTreeRange);
    const float cx = inside ? ux : 0.0f, cy = inside ? uy : 0.0f, cz = inside ? uz : 0.0f;
    const uint32_t qx = (uint32_t)__fmul_rn(cx, 2097152.0f), qy = (uint32_t)__fmul_rn(cy, 2097152.0f),
                   qz = (uint32_t)__fmul_rn(cz, 2097152.0f);
    u4[i] = make_float4(ux, uy, uz, hu);
    zt[i] = z[i];
    const int c = perm[i];
    key[c] = (spread3(qx) << 2) | (spread3(qy) << 1) | spread3(qz);
    val[c] = i;
  }
}

// ---- stable LSD radix sort of (key, value), 8-bit digits -------------------
// hist[d][tile]: count of digit d in each tile of kSortTile keys.
static __global__ void __launch_bounds__(kSortThreads)
radix_hist_kernel(const uint64_t* __restrict__ key, int n, int shift, int ntiles, unsigned* __restrict__ hist) {
  __shared__ unsigned hcount[256];
  hcount[threadIdx.x] = 0;
  __syncthreads();
  const int base = blockIdx.x * kSortTile;
  for (int r = 0; r < kSortRounds; ++r) {
    const int q = base + r * kSortThreads + threadIdx.x;
    if (q < n) atomicAdd(&hcount[(unsigned)(key[q] >> shift) & 255u], 1u);
  }
  __syncthreads();
  hist[(size_t)threadIdx.x * ntiles + blockIdx.x] = hcount[threadIdx.x];
}

// Exclusive scan of m counts (m a multiple of 4: 256 per sort tile) by one CTA, 4,096 at a time with
// a running sum; total (may be null) gets the sum. Every access is a coalesced 128-bit one (each
// thread walking a chunk of its own took 56 us for 32,768 counts).
static __global__ void __launch_bounds__(1024)
scan_exclusive_kernel(const unsigned* __restrict__ in, unsigned* __restrict__ out, int m, unsigned* total) {
  __shared__ unsigned part[32];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  auto load = [&](int k) { return k < m ? *reinterpret_cast<const uint4*>(in + k) : make_uint4(0, 0, 0, 0); };
  auto inclusive = [&](unsigned v) {  // over the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned t = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += t;
    }
    return v;
  };
  unsigned run = 0;
  uint4 v = load(4 * threadIdx.x);
  for (int base = 0; base < m; base += 4096) {
    const int k = base + 4 * threadIdx.x;
    const uint4 next = load(k + 4096);
    const unsigned s = v.x + v.y + v.z + v.w, i = inclusive(s);
    if (lane == 31) part[w] = i;
    __syncthreads();
    if (w == 0) part[lane] = inclusive(part[lane]);
    __syncthreads();
    const unsigned e = run + (w > 0 ? part[w - 1] : 0u) + i - s;
    if (k < m)
      *reinterpret_cast<uint4*>(out + k) = make_uint4(e, e + v.x, e + v.x + v.y, e + v.x + v.y + v.z);
    run += part[31];
    v = next;
    __syncthreads();
  }
  if (total && threadIdx.x == 0) *total = run;
}

// Stable scatter: the keys of a tile are taken in order, kSortThreads per
// round; within a round a key's rank among equal digits comes from its warp
// (match) and the warps before it, across rounds from a running count.
static __global__ void __launch_bounds__(kSortThreads)
radix_scatter_kernel(const uint64_t* __restrict__ kin, const int* __restrict__ vin, int n, int shift, int ntiles,
                     const unsigned* __restrict__ offs, uint64_t* __restrict__ kout, int* __restrict__ vout) {
  constexpr int kWarps = kSortThreads / 32;
  __shared__ unsigned run[256];
  __shared__ unsigned wcnt[kWarps][256];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  run[threadIdx.x] = offs[(size_t)threadIdx.x * ntiles + blockIdx.x];
  const unsigned lt = (1u << lane) - 1u;
  for (int r = 0; r < kSortRounds; ++r) {
    for (int k = 0; k < kWarps; ++k) wcnt[k][threadIdx.x] = 0;
    __syncthreads();
    const int q = blockIdx.x * kSortTile + r * kSortThreads + threadIdx.x;
    const bool valid = q < n;
    const uint64_t kv = valid ? kin[q] : 0ull;
    const int vv = valid ? vin[q] : 0;
    const unsigned dig = valid ? ((unsigned)(kv >> shift) & 255u) : 256u;
    const unsigned peers = __match_any_sync(0xffffffffu, dig);
    const unsigned rank = __popc(peers & lt);
    if (valid && rank == 0) wcnt[w][dig] = __popc(peers);
    __syncthreads();
    {
      unsigned acc = run[threadIdx.x];
      for (int k = 0; k < kWarps; ++k) {
        const unsigned cnt = wcnt[k][threadIdx.x];
        wcnt[k][threadIdx.x] = acc;
        acc += cnt;
      }
      run[threadIdx.x] = acc;
    }
    __syncthreads();
    if (valid) {
      const unsigned pos = wcnt[w][dig] + rank;
      kout[pos] = kv;
      vout[pos] = vv;
    }
    __syncthreads();
  }
}

// ---- level-by-level build ---------------------------------------------------
// Node records: link = (first child or -1, children, first, end sorted
// positions), geo = (centre, side) in root units, pre = key prefix.
// Thread per (active node, child digit): the child's sorted range. blk[CTA]: how many of the
// CTA's slots hold a child, and how many of these are active at the next level.
constexpr int kSlotThreads = 256;
static __global__ void __launch_bounds__(kSlotThreads)
tree_children_kernel(const int* __restrict__ active, int n_active, int level, int leaf,
                     const uint64_t* __restrict__ key, const int4* __restrict__ link,
                     const uint64_t* __restrict__ pre, int* __restrict__ cnt, int* __restrict__ beg,
                     int2* __restrict__ blk) {
  const int slot = blockIdx.x * blockDim.x + threadIdx.x;
  int ck = 0;
  if (slot < 8 * n_active) {
    const int node = active[slot >> 3], c = slot & 7;
    const int4 lk = link[node];
    const int sh = 3 * (kTreeDepth - 1 - level);
    const uint64_t target = (pre[node] << 3) | (uint64_t)c;
    int lo = lk.z, hi = lk.w;  // first q with key[q] >> sh >= target
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if ((key[mid] >> sh) < target) lo = mid + 1;
      else hi = mid;
    }
    int lo2 = lo, hi2 = lk.w;  // first q with key[q] >> sh > target
    while (lo2 < hi2) {
      const int mid = (lo2 + hi2) >> 1;
      if ((key[mid] >> sh) <= target) lo2 = mid + 1;
      else hi2 = mid;
    }
    ck = lo2 - lo;
    cnt[slot] = ck;
    beg[slot] = lo;
  }
  const int c1 = __syncthreads_count(ck > 0);
  const int c2 = __syncthreads_count(level + 1 < kTreeDepth && ck > leaf);
  if (threadIdx.x == 0) blk[blockIdx.x] = make_int2(c1, c2);
}

// Numbers the non-empty child slots (new nodes from id `base`, in slot order, so each
// parent's children are consecutive) and the next active nodes; writes the children, links the
// parents, and stores the two totals. Each CTA adds up the counts of the CTAs before it, a few
// hundred words from L2 (one CTA walking all slots took 65 us at the widest level of N = 262,144).
static __global__ void __launch_bounds__(kSlotThreads)
tree_link_kernel(const int* __restrict__ active, int n_active, int level, int leaf, int base,
                 const int* __restrict__ cnt, const int* __restrict__ beg, const int2* __restrict__ blk,
                 int4* __restrict__ link, float4* __restrict__ geo, uint64_t* __restrict__ pre,
                 int* __restrict__ next_active, int* __restrict__ totals) {
  constexpr int kWarps = kSlotThreads / 32;
  __shared__ int before1[kWarps], before2[kWarps], here1[kWarps], here2[kWarps];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int slot = blockIdx.x * blockDim.x + threadIdx.x;
  int b1 = 0, b2 = 0;
  for (int k = threadIdx.x; k < (int)blockIdx.x; k += kSlotThreads) {
    const int2 c = blk[k];
    b1 += c.x;
    b2 += c.y;
  }
  b1 = __reduce_add_sync(0xffffffffu, b1);
  b2 = __reduce_add_sync(0xffffffffu, b2);
  const int ck = slot < 8 * n_active ? cnt[slot] : 0;
  const bool child = ck > 0, deep = level + 1 < kTreeDepth && ck > leaf;
  const unsigned m1 = __ballot_sync(0xffffffffu, child), m2 = __ballot_sync(0xffffffffu, deep);
  if (lane == 0) {
    before1[w] = b1;
    before2[w] = b2;
    here1[w] = __popc(m1);
    here2[w] = __popc(m2);
  }
  __syncthreads();
  int p1 = __popc(m1 & ((1u << lane) - 1u)), p2 = __popc(m2 & ((1u << lane) - 1u));
#pragma unroll
  for (int k = 0; k < kWarps; ++k) {
    p1 += before1[k] + (k < w ? here1[k] : 0);
    p2 += before2[k] + (k < w ? here2[k] : 0);
  }
  if (child) {
    const float side = ldexpf(1.0f, -(level + 1));
    const int id = base + p1, bk = beg[slot];
    const uint64_t pf = (pre[active[slot >> 3]] << 3) | (uint64_t)(slot & 7);
    pre[id] = pf;
    link[id] = make_int4(-1, 0, bk, bk + ck);
    const uint32_t ix = compact3(pf >> 2), iy = compact3(pf >> 1), iz = compact3(pf);
    geo[id] = make_float4(__fmul_rn((float)ix + 0.5f, side), __fmul_rn((float)iy + 0.5f, side),
                          __fmul_rn((float)iz + 0.5f, side), side);
    if (deep) next_active[p2] = id;
  }
  if (slot < 8 * n_active && (slot & 7) == 0) {  // a node's eight slots lie in one warp
    const int node = active[slot >> 3];
    int4 lk = link[node];
    lk.x = base + p1;
    lk.y = __popc((m1 >> lane) & 0xffu);
    link[node] = lk;
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kSlotThreads - 1) {
    totals[0] = p1 + (child ? 1 : 0);
    totals[1] = p2 + (deep ? 1 : 0);
  }
}

// Moments of the nodes [n0, n1): a leaf sums its particles (sorted order), all leaves in one
// launch; then level by level from the deepest an inner node sums its children (FP64). mom = (M,
// sum m x, sum m y, sum m z'); hmax: largest h; hmf: largest hu.
template <bool LEAF>
__global__ void tree_moments_kernel(int n0, int n1, const int4* __restrict__ link,
                                           const int* __restrict__ sidx, const double* __restrict__ x,
                                           const double* __restrict__ y, const double* __restrict__ zt,
                                           const double* __restrict__ m, const double* __restrict__ h,
                                           const float4* __restrict__ u4, double4_32a* __restrict__ mom,
                                           double* __restrict__ hmax, float* __restrict__ hmf) {
  const int id = n0 + blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= n1) return;
  const int4 lk = link[id];
  if ((lk.y == 0) != LEAF) return;
  double M = 0.0, sx = 0.0, sy = 0.0, sz = 0.0, hm = 0.0;
  float hu = 0.0f;
  if (LEAF) {
    for (int q = lk.z; q < lk.w; ++q) {
      const int i = sidx[q];
      const double mi = m[i];
      M += mi;
      sx = fma(mi, x[i], sx);
      sy = fma(mi, y[i], sy);
      sz = fma(mi, zt[i], sz);
      hm = fmax(hm, h[i]);
      hu = fmaxf(hu, u4[i].w);
    }
  } else {
    for (int k = lk.x; k < lk.x + lk.y; ++k) {
      const double4_32a c = mom[k];
      M += c.x;
      sx += c.y;
      sy += c.z;
      sz += c.w;
      hm = fmax(hm, hmax[k]);
      hu = fmaxf(hu, hmf[k]);
    }
  }
  mom[id] = make_double4_32a(M, sx, sy, sz);
  hmax[id] = hm;
  hmf[id] = hu;
}

// Pseudo-particles of all nodes in the pair kernels' layout (periodic: z of
// the centre of mass shifted back by zeta into [0, L)).
static __global__ void tree_pack_kernel(int nn, const double4_32a* __restrict__ mom, const double* __restrict__ hmax,
                                        double zeta, double L, double invL, int periodic, float4* __restrict__ nA,
                                        float4* __restrict__ nB) {
  for (int id = blockIdx.x * blockDim.x + threadIdx.x; id < nn; id += gridDim.x * blockDim.x) {
    const double4_32a c = mom[id];
    double zc = c.w / c.x - zeta;
    if (periodic && zc < 0.0) zc += L;
    pack_one(c.y / c.x, c.z / c.x, zc, c.x, hmax[id], id, invL, __int_as_float(0x7f800000), nA, nB);
  }
}

// Particles in key order in the pair kernels' layout (coalesced leaf reads),
// with their tree-frame coordinates.
static __global__ void tree_gather_kernel(const float4* __restrict__ jA, const float4* __restrict__ jB,
                                          const float4* __restrict__ u4, const int* __restrict__ sidx, int n,
                                          float4* __restrict__ sA, float4* __restrict__ sB,
                                          float4* __restrict__ u4s) {
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
    const int i = sidx[q];
    sA[q] = jA[i];
    sB[q] = jB[i];
    u4s[q] = u4[i];
  }
}

// ---- walk ---------------------------------------------------------------------
// The opening test of one lane (FP32, exactly rounded, in the order written).
__device__ __forceinline__ bool tree_opens(const float4& u, const float4& g, float hm, const TreeCrit& C) {
  const float dx = __fsub_rn(u.x, g.x);
  const float dy = __fsub_rn(u.y, g.y);
  float dz = __fsub_rn(u.z, g.z);
  if (dz > C.hLu) dz = __fsub_rn(dz, C.Lu);
  else if (dz < -C.hLu) dz = __fadd_rn(dz, C.Lu);
  const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(dx, dx), __fmul_rn(dy, dy)), __fmul_rn(dz, dz));
  if (__fmul_rn(g.w, g.w) >= __fmul_rn(C.th2, d2)) return true;
  // far from the softening sum (with a margin for the rounding of both sides): no need of the root
  const float far = 0.8660254f * g.w + (u.w + hm);
  if (d2 > 1.0001f * far * far) return false;
  const float clear = __fsub_rn(__fsqrt_rn(d2), __fmul_rn(0.8660254f, g.w));
  return clear <= __fadd_rn(u.w, hm);
}

// A warp's interaction list, one array per word, so that one 64-bit load (the same address on
// every lane) yields two entries as a packed operand of pair2.cuh's two-pair forms.
struct TreeList {
  float xh[kWalkList], yh[kWalkList], zh[kWalkList], m[kWalkList];
  float xl[kWalkList], yl[kWalkList], zl[kWalkList], h[kWalkList];
  __device__ __forceinline__ void put(int k, const float4& a, const float4& b) {
    xh[k] = a.x;
    yh[k] = a.y;
    zh[k] = a.z;
    m[k] = a.w;
    xl[k] = b.x;
    yl[k] = b.y;
    zl[k] = b.z;
    h[k] = b.w;
  }
  __device__ __forceinline__ static u64 two(const float* v, int k) { return *reinterpret_cast<const u64*>(v + k); }
};
static_assert(kWalkList % 2 == 0, "an odd list is filled up by one entry");

// A lane's particle against the entries k and k + 1: separations and softening sums.
__device__ __forceinline__ void tree_separation(const I2& I, const TreeList& T, int k, bool periodic, Sep2& P) {
  P.dx = add2(sub2(I.xh, TreeList::two(T.xh, k)), sub2(I.xl, TreeList::two(T.xl, k)));
  P.dy = add2(sub2(I.yh, TreeList::two(T.yh, k)), sub2(I.yl, TreeList::two(T.yl, k)));
  const u64 zl = sub2(I.zl, TreeList::two(T.zl, k));
  const u64 d = sub2(I.zh, TreeList::two(T.zh, k)), r = dup(kRound23);
  P.dz = add2(periodic ? sub2(d, sub2(add2(d, r), r)) : d, zl);
  P.dr2 = fma2(P.dx, P.dx, mul2(P.dy, P.dy));
  P.hh = add2(I.h, TreeList::two(T.h, k));
}

// Pair forms of two list entries: image sums (SR, SZ).
// S1xR2: the correction-table tail over the infinite window; n0 = 4 in closed form, as the
// direct kernels take it (pair_sym.cuh), else near images and base one by one.
// RAW: the nearest-image table (n0 = 0), which holds the tail sums themselves.
template <int MODEL, bool RAW>
struct TreeTableForm {
  static constexpr bool periodic = true;
  const SurrConst& S;
  const TableTail& T;
  __device__ __forceinline__ void operator()(const Sep2& P, u64& SR, u64& SZ) const {
    const u64 ADZ = abs2(P.dz);
    Model2 M;
    model_stage2<MODEL, RAW, false>(P, ADZ, 0, S, M);
    float u0, v0, u1, v1;
    upk(M.u[0], u0, v0);
    upk(M.u[1], u1, v1);
    const float2 r = table_read(T, u0, u1), s = table_read(T, v0, v1);
    model_finish2<MODEL, RAW>(P, ADZ, 0, M, pk(r.x, s.x), pk(r.y, s.y), SR, SZ);
  }
};
// R^3 (eq. NewtonianForce): one image, the spline only when some lane is softened.
struct TreeR3Form {
  static constexpr bool periodic = false;
  __device__ __forceinline__ void operator()(const Sep2& P, u64& SR, u64& SZ) const {
    const u64 R2 = fma2(P.dz, P.dz, P.dr2), RI = rsq2(max2(R2, 1e-30f));
    SR = mul2(mul2(RI, RI), RI);
    if (any_less2(R2, mul2(P.hh, P.hh))) {
      const Soft2 s = soft2(P.hh);
      SR = spline_value_r2(R2, RI, SR, s.ih, s.nih, s.ih3);
    }
    SZ = mul2(P.dz, SR);
  }
};

// Packed sums of a lane: the two halves hold the even and the odd entries.
struct TreeSum {
  u64 x = 0, y = 0, z = 0, cx = 0, cy = 0, cz = 0;
};

// All lanes against the nl entries of the warp's list, two per step. A lane's own particle is
// among them: its separation is zero, so it adds exact zeros.
template <bool KAHAN, class Form>
__device__ __forceinline__ void tree_eval(const I2& I, TreeList& L, int nl, int lane, const Form& form, TreeSum& A) {
  if (nl & 1) {  // an odd list ends with a massless entry far off the axis
    if (lane == 0) L.put(nl, make_float4(4096.0f, 4096.0f, 0.0f, 0.0f), make_float4(0.0f, 0.0f, 0.0f, 0.0f));
    __syncwarp();
  }
#pragma unroll 1
  for (int k0 = 0; k0 < nl; k0 += 2 * STEPS_KAHAN_GROUP) {
    u64 gx = 0, gy = 0, gz = 0;
    const int ke = min(nl, k0 + 2 * STEPS_KAHAN_GROUP);
#pragma unroll 1
    for (int k = k0; k < ke; k += 2) {
      Sep2 P;
      tree_separation(I, L, k, Form::periodic, P);
      u64 SR, SZ;
      form(P, SR, SZ);
      const u64 m = TreeList::two(L.m, k), MS = mul2(m, SR);
      gx = fma2(P.dx, MS, gx);
      gy = fma2(P.dy, MS, gy);
      gz = fma2(m, SZ, gz);
    }
    acc2<KAHAN>(A.x, A.cx, gx);
    acc2<KAHAN>(A.y, A.cy, gy);
    acc2<KAHAN>(A.z, A.cz, gz);
  }
}

#ifndef STEPS_TREE_MIN_BLOCKS
// Co-resident CTAs per SM asked of the register allocator: 24 against 20 walk N = 262,144 in 7.48 against
// 7.54 ms, 400,000 in 12.3 against 13.3.
#define STEPS_TREE_MIN_BLOCKS (24 / STEPS_TREE_WARPS)
#endif

// One warp per group of 32 particles in key order (sA/sB, u4s: key order);
// out = [3][n] pair sums in internal order (sidx maps key order to internal).
// parts > 1: that many warps share a group's walk, each taking the subtrees of the tree's level kPartLevel
// whose number is `part` modulo parts (and part 0 what ends above that level), with its own sums
// out + 3 n part. A warp's walk takes milliseconds, so with a few warps per place on the GPU the last ones run
// nearly alone; the opened nodes above the level are tested by every part.
// FORM: S1xR2 with the near range n0 = 4, any other, or none (the nearest-image table), or the
// R^3 pair force (no images, no table).
enum TreeForm { kTreeInf4, kTreeInf, kTreeRaw, kTreeR3 };

#ifndef STEPS_TREE_PART_LEVEL
#define STEPS_TREE_PART_LEVEL 6
#endif
constexpr int kPartLevel = STEPS_TREE_PART_LEVEL, kMaxParts = 8;
// As many parts as make two and a half warps per place of `places`. Walk at N = 20,000 / 60,000 /
// 262,144, one part: 0.94 / 1.57 / 8.04 ms; two warps per place (8, 4, 1 parts) 0.60 / 1.36 / 7.93; four
// (8, 7, 2 parts) 0.60 / 1.54 / 7.54. Level 5 costs the same, 7 more at small N (0.84 at 20,000).
inline int walk_parts(int groups, int places) {
  return std::max(1, std::min(kMaxParts, (int)((5LL * places / 2 + groups - 1) / groups)));
}

template <bool KAHAN, int FORM>
__global__ void __launch_bounds__(kWalkWarps * 32, STEPS_TREE_MIN_BLOCKS)
tree_walk_kernel(const float4* __restrict__ sA, const float4* __restrict__ sB, const float4* __restrict__ u4s,
                 const int* __restrict__ sidx, int n, const int4* __restrict__ link, const float4* __restrict__ geo,
                 const float* __restrict__ hmf, const float4* __restrict__ nA, const float4* __restrict__ nB,
                 TreeCrit C, TableTail T, SurrConst S, int parts, double* __restrict__ out,
                 unsigned long long* __restrict__ inter, int* __restrict__ err) {
  __shared__ int stk[kWalkWarps][kWalkStack];
  __shared__ __align__(16) TreeList list[kWalkWarps];
  __shared__ float4 su[kWalkWarps][32];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gp = blockIdx.x * kWalkWarps + w, g = gp / parts, part = gp - g * parts;
  if (g * 32 >= n) return;  // the whole warp leaves; the walk uses warp-level synchronisation only
  const int q = g * 32 + lane;
  const bool valid = q < n;
  const int qc = min(q, n - 1);
  const float4 a = sA[qc], b = sB[qc];
  const I2 I{dup(a.x), dup(b.x), dup(a.y), dup(b.y), dup(a.z), dup(b.z), dup(b.w), 0};
  const int nvalid = min(32, n - g * 32);
  const float part_side = ldexpf(1.0f, -kPartLevel);
  int* st = stk[w];
  TreeList& L = list[w];
  TreeSum A;
  unsigned long long count = 0;
  bool overflow = false;
  su[w][lane] = u4s[qc];
  if (lane == 0) st[0] = 0;
  __syncwarp();
  // top nodes on the stack; the lanes `leaves` hold an opened leaf each (lf, particles lf.x .. lf.y)
  // and [p0, p1) is the one being listed; nl entries are listed. One place evaluates: a list without
  // room for 32 more, or the last one.
  int top = 1, nl = 0, p0 = 0, p1 = 0;
  unsigned leaves = 0;
  int2 lf = make_int2(0, 0);
  while (true) {
    const bool done = top == 0 && leaves == 0 && p0 == p1;
    if (nl > kWalkList - 33 || (done && nl > 0)) {
      __syncwarp();
      if constexpr (FORM == kTreeR3)
        tree_eval<KAHAN>(I, L, nl, lane, TreeR3Form{}, A);
      else
        tree_eval<KAHAN>(I, L, nl, lane, TreeTableForm<FORM == kTreeInf4 ? kModelInf4 : kModelInf, FORM == kTreeRaw>{S, T},
                         A);
      count += (unsigned long long)nl * nvalid;
      nl = 0;
      __syncwarp();
    }
    if (done) break;
    if (p0 < p1) {
      const int c = min(32, p1 - p0);
      if (lane < c) L.put(nl + lane, sA[p0 + lane], sB[p0 + lane]);
      nl += c;
      p0 += c;
      continue;
    }
    if (leaves) {
      const int l = __ffs(leaves) - 1;
      leaves &= leaves - 1;
      p0 = __shfl_sync(0xffffffffu, lf.x, l);
      p1 = __shfl_sync(0xffffffffu, lf.y, l);
      continue;
    }
    const int c = min(min(32, top), max(1, (kWalkStack - kWalkReserve - top) / 7));
    const bool mine = lane < c;
    const int node = mine ? st[top - 1 - lane] : 0;
    const float4 gm = geo[node];
    const int4 lk = link[node];
    const float hm = hmf[node];
    bool open = !mine;
    for (int k = 0; k < nvalid; ++k) {
      if (!open) open = tree_opens(su[w][k], gm, hm, C);
      if (__all_sync(0xffffffffu, open)) break;
    }
    top -= c;
    const unsigned lt = (1u << lane) - 1u;
    // with several parts, what ends above the level of the split belongs to the first
    const bool ours = mine && (parts == 1 || part == 0 || gm.w <= part_side);
    const unsigned take = __ballot_sync(0xffffffffu, ours && !open);
    if (ours && !open) L.put(nl + __popc(take & lt), nA[node], nB[node]);
    nl += __popc(take);
    const bool leaf = ours && open && lk.y == 0;
    leaves = __ballot_sync(0xffffffffu, leaf);
    lf = make_int2(lk.z, lk.w);
    // children, those of a lane's node together; at the level of the split this part's alone
    const bool split = parts > 1 && gm.w == 2.0f * part_side;
    int first = lk.x, step = 1, nc = mine && open ? lk.y : 0;
    if (split) {
      step = parts;
      first += (part - lk.x % parts + parts) % parts;
      nc = mine && open ? max(0, (lk.x + lk.y - first + parts - 1) / parts) : 0;
    }
    int at = nc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, at, o);
      if (lane >= o) at += t;
    }
    const int all = __shfl_sync(0xffffffffu, at, 31);
    at += top - nc;
    __syncwarp();  // every lane has read its node
    if (top + all > kWalkStack) {
      overflow = true;
      top = 0;
      leaves = 0;
      continue;
    }
    for (int k = 0; k < nc; ++k) st[at + k] = first + k * step;
    top += all;
    __syncwarp();
  }
  if (lane == 0) {
    atomicAdd(inter, count);
    if (overflow) atomicOr(err, kErrTreeStack);
  }
  if (valid) {
    const int i = sidx[q];
    out += 3 * (long long)n * part;
    double e, o;
    sum2<KAHAN>(A.x, A.cx, e, o);
    out[i] = e + o;
    sum2<KAHAN>(A.y, A.cy, e, o);
    out[(long long)n + i] = e + o;
    sum2<KAHAN>(A.z, A.cz, e, o);
    out[2 * (long long)n + i] = e + o;
  }
}

}  // namespace steps
