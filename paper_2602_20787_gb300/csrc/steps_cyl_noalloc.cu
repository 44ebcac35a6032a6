// Allocation-free pair accelerations (declared in include/steps_cyl.h as
// steps_cyl_pair_accel_noalloc).
//
// Some callers cannot allocate device memory: a host whose device memory is
// owned and budgeted by another allocator (a caching allocator or a fixed
// arena reserved at start-up), a loop that must not take cudaMalloc's implicit
// device-wide synchronisation, or a plug-in that is only allowed to allocate
// during its initialisation. For them this entry point evaluates the pair term
// with the same pair forms as a context does, but keeps every intermediate (the
// packed FP32 positions and the pair sums) in one file-scope __device__ array of
// fixed size. It never calls
// cudaMalloc, cudaFree or an allocating library routine. The call stays
// asynchronous, so it keeps no device error word: nothing would read it.
//
// The array exists once per device that loads this library and lives until the
// process exits. Host code cannot use its name as a device address: the address
// is obtained with cudaGetSymbolAddress once per device, with that device
// current, on the first call made on that device.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <mutex>

#include "steps_cyl.h"
#include "nbody_kernels.cuh"
#include "pair_sym.cuh"

using namespace steps;

namespace {

constexpr int kNoallocMaxN = STEPS_NOALLOC_MAX_N;
constexpr int kNoallocMaxCtas = STEPS_NOALLOC_MAX_CTAS;
constexpr int kNoallocMaxBlocks = (kNoallocMaxN + kBI - 1) / kBI;
// byte layout of the scratch array: packed jA | packed jB | partials
constexpr size_t kPackBytes = sizeof(float4) * (size_t)kNoallocMaxN;
constexpr size_t kPartBytes = sizeof(double) * 3 * kBI * (size_t)(kNoallocMaxBlocks + kNoallocMaxCtas);
constexpr size_t kScratchBytes = 2 * kPackBytes + kPartBytes;
static_assert(kScratchBytes == STEPS_NOALLOC_SCRATCH_BYTES, "scratch size must match the header");

__device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

// Each unordered pair is evaluated once where the fixed-point sums that this takes (two words,
// pair_sym.cuh) resolve the load. That needs the total mass and the largest one, the smallest softening and
// the extent, which the host cannot look at without waiting: the pack kernel reduces them on the
// device, its last CTA derives the scale, and the symmetric kernel or the row kernel takes the pairs; the
// other's CTAs return at once. (Derived by every CTA of the symmetric kernel, the scale cost the row route 20 us
// at N = 500, where its launch alone remains. N = 10,007, N_cut = 16, literal softening law: rows alone 730 us.)
// The record lies in the partials' last slot, which the row kernel's split never reaches.
constexpr int kPackThreads = 256;
constexpr int kPackParts = (kNoallocMaxN + kPackThreads - 1) / kPackThreads;
struct NoallocHead {
  unsigned long long hmin;  // bits of the smallest h; 0 when some h is not > 0
  unsigned long long rmax;  // bits of the largest (|x| + |y|) / L, no less than the distance from the axis
  unsigned long long mmax;  // bits of the largest |m|
  int err, sym;             // error bits of the symmetric kernel; whether it takes the pairs
  unsigned done;            // CTAs of the pack kernel that have finished
  unsigned massive;         // particles whose mass is not zero
  double scale;             // the sums' scale
  double mass[kPackParts];  // sums of |m| over each CTA of the pack kernel
};
constexpr size_t kHeadOffset = kScratchBytes - sizeof(double) * 3 * kBI;
static_assert(sizeof(NoallocHead) <= sizeof(double) * 3 * kBI, "the record takes one partial-sum slot");
static_assert(sizeof(unsigned long long) * 6 * kNoallocMaxN <= kPartBytes - sizeof(double) * 3 * kBI,
              "the fixed-point sums take the partials' place");

// The scale as the contexts choose it (2^57 over the bound on |S_i|), 0: none. By a whole warp, once
// every CTA's share is in the record (volatile: other CTAs wrote it).
__device__ __forceinline__ double noalloc_scale(const volatile NoallocHead* head, int parts, double L, int n_cut) {
  double M = 0.0;
  for (int k = threadIdx.x & 31; k < parts; k += 32) M += head->mass[k];
  for (int o = 16; o > 0; o >>= 1) M += __shfl_xor_sync(0xffffffffu, M, o);
  const double B = fix_bound(M, L / __longlong_as_double((long long)head->hmin), true);
  if (!(B >= 1e-290 && B < 1e270)) return 0.0;
  // one mass among massless particles has no sum of its own to resolve
  if (!fix_resolves(B, M, head->massive > 1 ? __longlong_as_double((long long)head->mmax) : 0.0,
                    2.0 * __longlong_as_double((long long)head->rmax), n_cut, kMaxSpreadF))
    return 0.0;
  const int S = 57 - (((__double2hiint(B) >> 20) & 0x7ff) - 1022);  // B < 2^(exponent + 1); |S| < 1,023
  return __hiloint2double((S + 1023) << 20, 0);
}

__global__ void __launch_bounds__(kPackThreads)
noalloc_pack_kernel(const double* __restrict__ x, const double* __restrict__ y, const double* __restrict__ z,
                    const double* __restrict__ m, const double* __restrict__ h, int n, double L, double invL, int n_cut,
                    float4* __restrict__ jA, float4* __restrict__ jB, unsigned long long* __restrict__ acc,
                    NoallocHead* head) {
  __shared__ double warp[kPackThreads / 32];
  __shared__ bool last;
  const int i = blockIdx.x * kPackThreads + threadIdx.x;
  double s = 0.0;
  unsigned long long hb = ~0ull, rb = 0, mb = 0;  // non-negative doubles order like their bits, NaN above all
  if (i < n) {
    pack_one(x[i], y[i], z[i], m[i], h[i], i, invL, kPackCap, jA, jB);
    for (int c = 0; c < 6; ++c) acc[c * (size_t)n + i] = 0;
    s = fabs(m[i]);
    hb = h[i] > 0.0 ? (unsigned long long)__double_as_longlong(h[i]) : 0ull;
    rb = (unsigned long long)__double_as_longlong((fabs(x[i]) + fabs(y[i])) * invL);
    mb = (unsigned long long)__double_as_longlong(s);
  }
  const unsigned massive = __popc(__ballot_sync(0xffffffffu, mb != 0));
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_down_sync(0xffffffffu, s, o);
    hb = min(hb, __shfl_down_sync(0xffffffffu, hb, o));
    rb = max(rb, __shfl_down_sync(0xffffffffu, rb, o));
    mb = max(mb, __shfl_down_sync(0xffffffffu, mb, o));
  }
  if ((threadIdx.x & 31) == 0) {
    warp[threadIdx.x >> 5] = s;
    atomicMin(&head->hmin, hb);
    atomicMax(&head->rmax, rb);
    atomicMax(&head->mmax, mb);
    atomicAdd(&head->massive, massive);
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kPackThreads / 32; ++w) t += warp[w];
    head->mass[blockIdx.x] = t;
    __threadfence();
    last = atomicAdd(&head->done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (last && threadIdx.x < 32) {
    __threadfence();
    const double scale = noalloc_scale(head, gridDim.x, L, n_cut);
    if (threadIdx.x == 0) {
      head->scale = scale;
      head->sym = scale > 0.0;
    }
  }
}

template <bool KAHAN, bool LINE>
__global__ void __launch_bounds__(kSymThreads, STEPS_SYM_MIN_BLOCKS)
noalloc_sym_kernel(const float4* __restrict__ jA, const float4* __restrict__ jB, int n, int n_cut, int NB, int tpb,
                   int sp, long long U, int C, unsigned long long* __restrict__ acc, NoallocHead* __restrict__ head) {
  __shared__ SymShared<KAHAN> sh;
  const double scale = head->scale;
  if (!(scale > 0.0)) return;
  const float f = scale <= ldexp(1.0, kMaxFixExpF) && scale >= ldexp(1.0, -kMaxFixExpF) ? (float)scale : 0.0f;
  sym_stream_k<KAHAN, true, KAHAN>(jA, jB, n, NB, tpb, sp, 0, U, C, sh,
                            FixAcc{acc, n, scale, f, &head->err, 0, 0, 0, 0, acc + 3 * (size_t)n},
                            PlainForm<LINE, false>{n_cut, (float)n_cut});
}

// Accelerations from either kernel's sums. A sum beyond the fixed-point range can only come from a
// position that is not finite, whose pairs with every particle give NaN.
__global__ void noalloc_finalize_kernel(const unsigned long long* __restrict__ acc, const double* __restrict__ part,
                                        const NoallocHead* __restrict__ head, int n, int NT, long long U, int C,
                                        double pair_scale, double* __restrict__ ax, double* __restrict__ ay,
                                        double* __restrict__ az) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double s[3] = {0.0, 0.0, 0.0};
  if (head->sym) {
    const double inv = 1.0 / head->scale;
    for (int q = 0; q < 3; ++q) {
      const size_t o = (size_t)q * n + i;
      s[q] = head->err ? __longlong_as_double(0x7ff8000000000000LL) : fix_sum(acc[o], acc + 3 * (size_t)n + o, inv);
    }
  } else {
    row_sums(part, i, NT, U, C, s[0], s[1], s[2]);
  }
  ax[i] = pair_scale * s[0];
  ay[i] = pair_scale * s[1];
  az[i] = pair_scale * s[2];
}

struct DeviceScratch {
  unsigned char* base = nullptr;  // device address of g_noalloc_scratch on this device
  int ctas = 0;                   // co-resident CTAs of the row kernel (capped)
  int sms = 0, sym_ctas = 0;      // SMs; co-resident CTAs of the symmetric kernel
  bool ready = false;
};

constexpr int kMaxDevices = 64;
DeviceScratch g_dev[kMaxDevices];
std::mutex g_mutex;

// Failures are reported by the status code alone (the message text names the
// cause for a reader of this file).
inline int noalloc_fail(int code, const char* /*why*/) { return code; }

// A runtime call of this entry point failed: clear the error it left as the
// thread's last error, unless an error from the caller's earlier work was
// already pending when the call began (that one stays for the caller to see).
inline int noalloc_cuda_fail(cudaError_t pending, const char* why) {
  if (pending == cudaSuccess) cudaGetLastError();
  return noalloc_fail(STEPS_ECUDA, why);
}

// Set-up for the current device (called with that device current).
int setup_device(int dev, cudaError_t pending, DeviceScratch** out) {
  std::lock_guard<std::mutex> lock(g_mutex);
  DeviceScratch& d = g_dev[dev];
  if (!d.ready) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess)
      return noalloc_cuda_fail(pending, "cudaGetSymbolAddress of the scratch array failed");
    int sms = 0, occ = 0, socc = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&socc, noalloc_sym_kernel<true, true>, kSymThreads, 0) !=
            cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, pair_row_kernel<true, true>, kPairThreads, 0) != cudaSuccess)
      return noalloc_cuda_fail(pending, "device query failed");
    d.base = static_cast<unsigned char*>(ptr);
    d.ctas = std::max(1, std::min(kNoallocMaxCtas, sms * std::max(occ, 1)));
    d.sms = sms;
    d.sym_ctas = sms * std::max(socc, 1);
    d.ready = true;
  }
  *out = &d;
  return STEPS_OK;
}

// True when p is device memory the kernels on device dev may dereference: an
// allocation of that device (cudaMalloc, a pool, VMM) or managed memory. Host
// memory, pinned or not, and another device's memory are refused.
// cudaPointerGetAttributes only reads the driver's records; it allocates nothing.
bool on_device(const void* p, int dev, cudaError_t pending) {
  cudaPointerAttributes at{};
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    if (pending == cudaSuccess) cudaGetLastError();
    return false;
  }
  if (at.type == cudaMemoryTypeManaged) return true;
  return at.type == cudaMemoryTypeDevice && at.device == dev;
}

}  // namespace

extern "C" int steps_cyl_pair_accel_noalloc(int64_t n, const double* x, const double* y, const double* z,
                                            const double* m, const double* h, double G, double L, int32_t n_cut,
                                            int32_t precision, double* ax, double* ay, double* az, void* stream) {
  if (n < 2 || n > kNoallocMaxN) return noalloc_fail(STEPS_EINVAL, "n must be in [2, STEPS_NOALLOC_MAX_N]");
  if (!x || !y || !z || !m || !h || !ax || !ay || !az) return noalloc_fail(STEPS_EINVAL, "NULL array");
  if (!(G > 0) || !(L > 0)) return noalloc_fail(STEPS_EINVAL, "G and L must be > 0");
  if (n_cut < 1 || n_cut > 4096) return noalloc_fail(STEPS_EINVAL, "n_cut must be in [1, 4096]");
  if (precision != STEPS_FP32_KAHAN && precision != STEPS_FP32_PLAIN)
    return noalloc_fail(STEPS_EINVAL, "precision must be STEPS_FP32_KAHAN or STEPS_FP32_PLAIN");
  const cudaError_t pending = cudaPeekAtLastError();
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return noalloc_cuda_fail(pending, "no usable current device");
  if (dev < 0 || dev >= kMaxDevices) return noalloc_fail(STEPS_ECUDA, "device ordinal beyond the table");
  const void* arrays[8] = {x, y, z, m, h, ax, ay, az};
  for (const void* p : arrays)
    if (!on_device(p, dev, pending))
      return noalloc_fail(STEPS_EINVAL, "every array must be device memory of the current device");
  DeviceScratch* d = nullptr;
  int rc = setup_device(dev, pending, &d);
  if (rc) return rc;

  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int nn = (int)n;
  float4* jA = reinterpret_cast<float4*>(d->base);
  float4* jB = reinterpret_cast<float4*>(d->base + kPackBytes);
  double* part = reinterpret_cast<double*>(d->base + 2 * kPackBytes);
  const int NB = (nn + kBI - 1) / kBI;
  const RowSplit row = row_split(NB, nn, d->ctas);
  const double invL = 1.0 / L;

  // every byte of the scratch array this call reads, it writes first: the record, the packed
  // positions and the cleared sums here, or each stream-K partial slot whole, before the
  // finalize kernel reads it
  NoallocHead* head = reinterpret_cast<NoallocHead*>(d->base + kHeadOffset);
  unsigned long long* acc = reinterpret_cast<unsigned long long*>(part);
  const int parts = (nn + kPackThreads - 1) / kPackThreads;
  cudaMemsetAsync(&head->hmin, 0xff, sizeof head->hmin, st);
  cudaMemsetAsync(&head->rmax, 0, offsetof(NoallocHead, scale) - offsetof(NoallocHead, rmax), st);
  noalloc_pack_kernel<<<parts, kPackThreads, 0, st>>>(x, y, z, m, h, nn, L, invL, n_cut, jA, jB, acc, head);
  const bool kahan = precision == STEPS_FP32_KAHAN;
  int tpb, sp;
  sym_split(NB, d->sms, true, tpb, sp);
  const long long SU = (long long)NB * (NB + 1) / 2 * tpb * sp;
  const int SC = (int)std::min<long long>(SU, 32LL * d->sym_ctas);
  auto sym = line_form_rows(n_cut) ? (kahan ? noalloc_sym_kernel<true, true> : noalloc_sym_kernel<false, true>)
                              : (kahan ? noalloc_sym_kernel<true, false> : noalloc_sym_kernel<false, false>);
  sym<<<SC, kSymThreads, 0, st>>>(jA, jB, nn, n_cut, NB, tpb, sp, SU, SC, acc, head);
  auto kernel = line_form_rows(n_cut) ? (kahan ? pair_row_kernel<true, true> : pair_row_kernel<false, true>)
                                 : (kahan ? pair_row_kernel<true, false> : pair_row_kernel<false, false>);
  kernel<<<row.C, kPairThreads, 0, st>>>(jA, jB, nn, n_cut, row.U, row.NT, row.jt, row.C, part, 0, &head->sym);
  const int ft = particle_threads(nn);
  noalloc_finalize_kernel<<<(nn + ft - 1) / ft, ft, 0, st>>>(acc, part, head, nn, row.NT, row.U, row.C, -G * invL * invL, ax, ay,
                                                             az);
  // a launch failure replaces the thread's last error; one equal to the error
  // pending before the call is taken as the caller's, which stays in place
  const cudaError_t after = cudaPeekAtLastError();
  if (after != cudaSuccess && after != pending) return noalloc_cuda_fail(pending, "a kernel launch failed");
  return STEPS_OK;
}
