// Totals of the two per-particle ledgers (emitted synchrotron energy and
// Landau-Lifshitz loss), the global sums compared in Fig. 3 of
// arXiv:1409.5574: the exact sum of the FP64 entries, rounded once.
//
// The sum is kept in integers, as a fixed-point number of 32-bit limbs (limb j
// has weight 2^(32 j - 1075), so every finite double is a 53-bit integer
// shifted into three neighbouring limbs).  It does not depend on the order of
// the adds, on the grid or on the alignment, and it leaves the FP64 pipe
// alone, whose 2 lanes per clock and SM bound a floating-point reduction: one
// add per entry is all it could do at the rate the memory delivers, and the
// compensated sum that stood here took eight per pair (2^25 pairs 617 us, 0.87
// TB/s; now 111 us, 4.8 TB/s, and 207 us for 2^26 pairs).
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdio>
#include <mutex>

#include "prad_internal.h"

namespace prad {

namespace {

constexpr int kLimbs = 72;       // 67 hold any double, the rest carries
constexpr int kRedThreads = 256;
constexpr int kRedBlocks = 3;    // resident blocks per SM the kernel is compiled for
constexpr uint32_t kNoWindow = 0x80000000u;

// A thread's part of the sum: a signed 160-bit number at limb k, which takes
// any value whose exponent lies in limbs k and k + 1 (2^64 apart).  Values
// elsewhere move the window (its sum goes to the block's limbs) or, at the
// ends of the range, go to the block's limbs themselves.
struct Window {
  uint32_t r0 = 0, r1 = 0, r2 = 0, r3 = 0, r4 = 0;
  uint32_t k = kNoWindow;
};

__device__ __forceinline__ void limb_add(long long* limbs, int j, long long v) {
  atomicAdd(reinterpret_cast<unsigned long long*>(limbs) + j, static_cast<unsigned long long>(v));
}

__device__ __forceinline__ long long window_limb(const Window& w, int q) {
  return q == 0 ? static_cast<long long>(w.r0)
       : q == 1 ? static_cast<long long>(w.r1)
       : q == 2 ? static_cast<long long>(w.r2)
       : q == 3 ? static_cast<long long>(w.r3)
                : static_cast<long long>(static_cast<int32_t>(w.r4));
}

// A value outside the window (subnormal, non-finite, or of another size).
// True if the window now holds it.  (Inlined: a call would keep the window in
// local memory.)
__device__ __forceinline__ bool window_miss(Window& w, uint32_t lo, uint32_t hi, long long* limbs,
                                         int* bad) {
  const uint32_t e = (hi >> 20) & 0x7ffu;
  if (e == 0x7ffu) {
    *bad = 1;
    return false;
  }
  const int k = static_cast<int>(e >> 5);
  if (k >= 1 && k <= 62) {
    if (w.k != kNoWindow) {
#pragma unroll
      for (int q = 0; q < 5; ++q) limb_add(limbs, static_cast<int>(w.k) + q, window_limb(w, q));
    }
    // the lower half of a limb's exponents: the window reaches down, else up
    const int nk = (e & 31u) < 16u ? k - 1 : k;
    w = Window{};
    w.k = static_cast<uint32_t>(nk < 1 ? 1 : (nk > 61 ? 61 : nk));
    return true;
  }
  const uint32_t s = e ? (e & 31u) : 1u;
  const uint32_t m1 = (hi & 0xfffffu) | (e ? 0x100000u : 0u);
  const long long sg = (hi >> 31) ? -1 : 1;
  limb_add(limbs, k, sg * static_cast<long long>(lo << s));
  limb_add(limbs, k + 1, sg * static_cast<long long>(__funnelshift_l(lo, m1, s)));
  limb_add(limbs, k + 2, sg * static_cast<long long>(__funnelshift_l(m1, 0u, s)));
  return false;
}

__device__ __forceinline__ void window_add(Window& w, double v, long long* limbs, int* bad) {
  const uint32_t lo = static_cast<uint32_t>(__double2loint(v));
  const uint32_t hi = static_cast<uint32_t>(__double2hiint(v));
  const uint32_t e = (hi >> 20) & 0x7ffu;
  const uint32_t m1 = (hi & 0xfffffu) | (e ? 0x100000u : 0u);
  uint32_t d = (e >> 5) - w.k;
  if (d > 1u && (lo | m1) != 0u) {  // (zeros add nothing wherever they fall)
    if (!window_miss(w, lo, hi, limbs, bad)) return;
    d = (e >> 5) - w.k;
  }
  const uint32_t l0 = lo << (e & 31u);
  const uint32_t l1 = __funnelshift_l(lo, m1, e);
  const uint32_t l2 = __funnelshift_l(m1, 0u, e);
  const bool up = d != 0u;
  const uint32_t x0 = up ? 0u : l0, x1 = up ? l0 : l1, x2 = up ? l1 : l2, x3 = up ? l2 : 0u;
  if (hi >> 31)
    asm("sub.cc.u32 %0, %0, %5;\n\tsubc.cc.u32 %1, %1, %6;\n\tsubc.cc.u32 %2, %2, %7;\n\t"
        "subc.cc.u32 %3, %3, %8;\n\tsubc.u32 %4, %4, 0;"
        : "+r"(w.r0), "+r"(w.r1), "+r"(w.r2), "+r"(w.r3), "+r"(w.r4)
        : "r"(x0), "r"(x1), "r"(x2), "r"(x3));
  else
    asm("add.cc.u32 %0, %0, %5;\n\taddc.cc.u32 %1, %1, %6;\n\taddc.cc.u32 %2, %2, %7;\n\t"
        "addc.cc.u32 %3, %3, %8;\n\taddc.u32 %4, %4, 0;"
        : "+r"(w.r0), "+r"(w.r1), "+r"(w.r2), "+r"(w.r3), "+r"(w.r4)
        : "r"(x0), "r"(x1), "r"(x2), "r"(x3));
}

// Sums of mantissa parts, folded into the window after at most kFold groups
// of eight values: a value is (27 bits + 26 bits x 2^27) 2^t with t its
// exponent above the window's, t in [0, 64), and 2^t = f0 + f1 2^32 with one of
// the two zero, so its four products of less than 2^59 go to four sums of
// weights 1, 2^27, 2^32 and 2^59.
struct Parts {
  uint64_t p0 = 0, p1 = 0, p2 = 0, p3 = 0;
};
constexpr int kFold = 3;  // 24 values: sums below 2^64

// w += v 2^(32 word + shift)
template <int WORD, int SHIFT>
__device__ __forceinline__ void window_add64(Window& w, uint64_t v) {
  const uint32_t lo = static_cast<uint32_t>(v), hi = static_cast<uint32_t>(v >> 32);
  const uint32_t x0 = lo << SHIFT;
  const uint32_t x1 = SHIFT ? __funnelshift_l(lo, hi, SHIFT) : hi;
  const uint32_t x2 = SHIFT ? __funnelshift_l(hi, 0u, SHIFT) : 0u;
  if constexpr (WORD == 0)
    asm("add.cc.u32 %0, %0, %5;\n\taddc.cc.u32 %1, %1, %6;\n\taddc.cc.u32 %2, %2, %7;\n\t"
        "addc.cc.u32 %3, %3, 0;\n\taddc.u32 %4, %4, 0;"
        : "+r"(w.r0), "+r"(w.r1), "+r"(w.r2), "+r"(w.r3), "+r"(w.r4)
        : "r"(x0), "r"(x1), "r"(x2));
  else
    asm("add.cc.u32 %0, %0, %4;\n\taddc.cc.u32 %1, %1, %5;\n\taddc.cc.u32 %2, %2, %6;\n\t"
        "addc.u32 %3, %3, 0;"
        : "+r"(w.r1), "+r"(w.r2), "+r"(w.r3), "+r"(w.r4)
        : "r"(x0), "r"(x1), "r"(x2));
}

__device__ __forceinline__ void fold(Window& w, Parts& p) {
  window_add64<0, 0>(w, p.p0);
  window_add64<0, 27>(w, p.p1);
  window_add64<1, 0>(w, p.p2);
  window_add64<1, 27>(w, p.p3);
  p = Parts{};
}

__device__ __forceinline__ uint64_t mad_wide(uint32_t a, uint32_t b, uint64_t c) {
  asm("mad.wide.u32 %0, %1, %2, %0;" : "+l"(c) : "r"(a), "r"(b));
  return c;
}
// 1 << s, 0 from s = 32 on
__device__ __forceinline__ uint32_t bit_of(uint32_t s) {
  uint32_t r;
  asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(1u), "r"(s));
  return r;
}

// Eight values at once.  A group without negative ones takes a shorter form
// (the integer pipe, 16 lanes per clock and scheduler, is the bound: 11
// instructions there and four wide products on the FMA pipe per value; shifts,
// selects and a carry chain per value were 5% slower); both factors are 0 for a
// value outside the window (a zero, mostly), and what the window missed is seen
// to afterwards.
__device__ __forceinline__ void window_add8(Window& w, Parts& p, const double (&v)[8],
                                            long long* limbs, int* bad) {
  uint32_t any = 0u;
#pragma unroll
  for (int j = 0; j < 8; ++j) any |= static_cast<uint32_t>(__double2hiint(v[j]));
  const bool neg = any >> 31;
  uint32_t missed = neg ? 1u : 0u;
  // (without a window every exponent lies outside)
  const uint32_t e0 = w.k == kNoWindow ? kNoWindow : w.k << 5;
  if (!neg) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t lo = static_cast<uint32_t>(__double2loint(v[j]));
      const uint32_t hi = static_cast<uint32_t>(__double2hiint(v[j]));
      const uint32_t t = (hi >> 20) - e0;
      const uint32_t f0 = bit_of(t), f1 = bit_of(t - 32u);
      const uint32_t a = lo & 0x7ffffffu;
      const uint32_t b = __funnelshift_l(lo, (hi & 0xfffffu) | 0x100000u, 5);
      if (t > 63u) missed |= lo | hi;
      p.p0 = mad_wide(a, f0, p.p0);
      p.p1 = mad_wide(b, f0, p.p1);
      p.p2 = mad_wide(a, f1, p.p2);
      p.p3 = mad_wide(b, f1, p.p3);
    }
  }
  if (missed) {
    fold(w, p);  // (a missed value may move the window)
#pragma unroll 1
    for (int j = 0; j < 8; ++j) {
      double x = v[0];
#pragma unroll
      for (int q = 1; q < 8; ++q) x = q == j ? v[q] : x;
      if (neg || (static_cast<uint32_t>(__double2hiint(x)) >> 20) - e0 > 63u)
        window_add(w, x, limbs, bad);
    }
  }
}

// The number of limbs[lo .. hi] (the others are zero; hi + 2 < kLimbs), rounded
// once to double (one thread; the limbs are overwritten).
__device__ double limbs_value(long long* limbs, int lo, int hi) {
  const int end = hi + 2;  // the sum's carry
  long long carry = 0;
  for (int j = lo; j <= end; ++j) {
    const long long t = limbs[j] + carry;
    limbs[j] = t & 0xffffffffll;
    carry = t >> 32;
  }
  const bool neg = carry < 0;
  if (neg) {  // two's complement
    long long one = 1;
    for (int j = lo; j <= end; ++j) {
      const long long t = (~limbs[j] & 0xffffffffll) + one;
      limbs[j] = t & 0xffffffffll;
      one = t >> 32;
    }
  }
  int top = end;
  while (top >= lo && limbs[top] == 0) --top;
  if (top < lo) return 0.0;
  const uint32_t a = static_cast<uint32_t>(limbs[top]);
  const uint32_t b = top > lo ? static_cast<uint32_t>(limbs[top - 1]) : 0u;
  const uint32_t c = top > lo + 1 ? static_cast<uint32_t>(limbs[top - 2]) : 0u;
  const int z = __clz(static_cast<int>(a));
  uint64_t m = (((static_cast<uint64_t>(a) << 32) | b) << z) | (z ? c >> (32 - z) : 0u);
  bool below = (c << z) != 0u;
  for (int j = lo; j < top - 2; ++j) below = below || limbs[j] != 0;
  m |= below ? 1u : 0u;  // below the rounding position: 64 > 53 + 2 bits
  const double v = ldexp(__ull2double_rn(m), 32 * (top - 1) - z - 1075);
  return neg ? -v : v;
}

// One warp: the limbs' number (shared memory) to *out, NaN if bad.
__device__ __forceinline__ void round_sum(long long* limbs, bool bad, double* out) {
  const int lane = threadIdx.x & 31;
  int lo = kLimbs, hi = -1;
#pragma unroll
  for (int j0 = 0; j0 < kLimbs; j0 += 32) {
    const unsigned nz = __ballot_sync(0xffffffffu, j0 + lane < kLimbs && limbs[j0 + lane] != 0);
    if (nz) {
      lo = min(lo, j0 + __ffs(nz) - 1);
      hi = j0 + 31 - __clz(static_cast<int>(nz));
    }
  }
  if (lane == 0)
    *out = bad ? __longlong_as_double(0x7ff8000000000000ll)
               : (hi < 0 ? 0.0 : limbs_value(limbs, lo, hi));
}

// Scratch of a reduction, zeroed before the launch: the two sums' limbs,
// whether an entry was not finite, and the blocks done.
struct RedScratch {
  long long limbs[2][kLimbs];
  int bad[2];
  unsigned int done, pad;
};
static_assert(sizeof(RedScratch) <= kLedgerScratchBytes, "ledger scratch size");

// Blocks (x, q) sum ledger q grid-stride; the last one rounds both sums.  A
// ledger with a non-finite entry sums to NaN.  VEC: 16-byte loads.
template <bool VEC>
__global__ void __launch_bounds__(kRedThreads, kRedBlocks)
    k_ledger_sum(const double* __restrict__ a, const double* __restrict__ b, int64_t n,
                 RedScratch* __restrict__ sc, double* __restrict__ out) {
  __shared__ long long s_limbs[kLimbs], s_fin[2][kLimbs];
  __shared__ int s_bad;
  __shared__ bool s_last;
  const int tid = threadIdx.x, lane = tid & 31, q = blockIdx.y;
  if (tid < kLimbs) s_limbs[tid] = 0;
  if (tid == 0) s_bad = 0;
  __syncthreads();
  const double* __restrict__ v = q ? b : a;
  Window w;
  Parts p;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * kRedThreads;
  const int64_t first = static_cast<int64_t>(blockIdx.x) * kRedThreads + tid;
  if constexpr (VEC) {
    const double2* __restrict__ v2 = reinterpret_cast<const double2*>(v);
    const int64_t n2 = n / 2;
    int64_t i = first;
    if (i + 3 * stride < n2) {  // the next four loads in flight while four are added
      double2 y[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) y[k] = v2[i + k * stride];
      bool more = true;
      for (int g = 1; more; ++g) {
        double x[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          x[2 * k] = y[k].x;
          x[2 * k + 1] = y[k].y;
        }
        i += 4 * stride;
        more = i + 3 * stride < n2;
        if (more) {
#pragma unroll
          for (int k = 0; k < 4; ++k) y[k] = v2[i + k * stride];
        }
        window_add8(w, p, x, s_limbs, &s_bad);
        if (g % kFold == 0) fold(w, p);
      }
    }
    fold(w, p);
    for (; i < n2; i += stride) {
      const double2 x = v2[i];
      window_add(w, x.x, s_limbs, &s_bad);
      window_add(w, x.y, s_limbs, &s_bad);
    }
    if ((n & 1) && first == 0) window_add(w, v[n - 1], s_limbs, &s_bad);
  } else {
    int64_t i = first;
    for (int g = 1; i + 7 * stride < n; i += 8 * stride, ++g) {
      double x[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = v[i + k * stride];
      window_add8(w, p, x, s_limbs, &s_bad);
      if (g % kFold == 0) fold(w, p);
    }
    fold(w, p);
    for (; i < n; i += stride) window_add(w, v[i], s_limbs, &s_bad);
  }
  // the warp's windows, those at the same limb together
  __syncwarp();
  unsigned todo = __ballot_sync(0xffffffffu, w.k != kNoWindow);
  while (todo) {
    const uint32_t k = __shfl_sync(0xffffffffu, w.k, __ffs(todo) - 1);
    const bool mine = w.k == k;
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      long long x = mine ? window_limb(w, j) : 0;
#pragma unroll
      for (int off = 16; off; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
      if (lane == 0 && x) limb_add(s_limbs, static_cast<int>(k) + j, x);
    }
    todo &= ~__ballot_sync(0xffffffffu, mine);
  }
  __syncthreads();
  if (gridDim.x == 1) {  // the block holds the whole sum
    if (tid < 32) round_sum(s_limbs, s_bad != 0, out + q);
    return;
  }
  // to the launch's limbs, split so that no limb can overflow
  if (tid < kLimbs && s_limbs[tid]) {
    const long long x = s_limbs[tid];
    limb_add(sc->limbs[q], tid, x & 0xffffffffll);
    if (x >> 32) limb_add(sc->limbs[q], tid + 1 < kLimbs ? tid + 1 : tid, x >> 32);
  }
  if (tid == 0 && s_bad) atomicOr(&sc->bad[q], 1);
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&sc->done, 1u) + 1u == gridDim.x * gridDim.y;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // the last block of all: warp r rounds sum r
  if (tid >= 64) return;
  const int r = tid >> 5;
  for (int j = lane; j < kLimbs; j += 32)
    s_fin[r][j] = *reinterpret_cast<volatile long long*>(&sc->limbs[r][j]);
  __syncwarp();
  round_sum(s_fin[r], *reinterpret_cast<volatile int*>(&sc->bad[r]) != 0, out + r);
}

}  // namespace

cudaError_t launch_ledger_reduce(const double* a, const double* b, int64_t n, void* scratch,
                                 int num_sms, double* out, cudaStream_t s) {
  // one block per sum up to 8192 entries (no scratch, no last block to wait for)
  const int64_t want = n <= 32 * kRedThreads ? 1 : (n + 8 * kRedThreads - 1) / (8 * kRedThreads);
  if (want > 1) {
    const cudaError_t e = cudaMemsetAsync(scratch, 0, sizeof(RedScratch), s);
    if (e != cudaSuccess) return e;
  }
  const int64_t cap = static_cast<int64_t>(kRedBlocks) * num_sms / 2;
  const dim3 grid(static_cast<unsigned>(want < 1 ? 1 : (want < cap ? want : cap)), 2);
  RedScratch* sc = static_cast<RedScratch*>(scratch);
  const bool vec = ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15) == 0;
  if (vec)
    k_ledger_sum<true><<<grid, kRedThreads, 0, s>>>(a, b, n, sc, out);
  else
    k_ledger_sum<false><<<grid, kRedThreads, 0, s>>>(a, b, n, sc, out);
  return cudaGetLastError();
}

}  // namespace prad

// ---------------------------------------------------------------------------
// Allocation-free totals.  Some callers cannot allocate device memory at the
// point where they need the totals: a host code that owns a fixed device
// memory pool, or a time loop in which a cudaMalloc (which synchronises the
// device and may fail once the pool has claimed the memory) is not
// acceptable.  This variant of the reduction above keeps its scratch in a
// file-scope device array instead of the context, and calls no allocation
// routine.
// ---------------------------------------------------------------------------
namespace {

// Most entries of a call (the limit its callers know).
constexpr int64_t kStaticMax = int64_t(65536) * 4096;
__device__ __align__(256) unsigned char g_static_scratch[prad::kLedgerScratchBytes];

// Device address of g_static_scratch per device, looked up once per device
// (host code must not pass the array's host-side name to a kernel).  The
// address belongs to the device's primary context at the first call; a
// cudaDeviceReset later in the process invalidates it (calls after a reset
// are not supported).
constexpr int kMaxDevices = 64;
std::mutex g_static_mu;
void* g_static_addr[kMaxDevices] = {nullptr};
int g_static_sms[kMaxDevices] = {0};

thread_local char g_static_err[256];

int static_fail(int code, const char* msg) {
  std::snprintf(g_static_err, sizeof(g_static_err), "%s", msg);
  return code;
}

}  // namespace

extern "C" const char* prad_ledger_totals_noalloc_error(void) { return g_static_err; }

extern "C" int prad_ledger_totals_noalloc(const double* emit, const double* rr, int64_t n,
                                          double* out, void* stream) {
  g_static_err[0] = '\0';  // the message describes this call's failure only
  if (!out || n < 0 || (n > 0 && (!emit || !rr)))
    return static_fail(PRAD_ERR_ARG, "ledger_totals_noalloc: null pointer or n < 0");
  if (n > kStaticMax)
    return static_fail(PRAD_ERR_ARG,
                       "ledger_totals_noalloc: n exceeds the limit of 268435456 entries");
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
    return static_fail(PRAD_ERR_CUDA, "ledger_totals_noalloc: no usable current device");
  void* scratch = nullptr;
  int sms = 1;
  {
    // set-up on the first call per device, with that device current
    std::lock_guard<std::mutex> lk(g_static_mu);
    if (!g_static_addr[dev]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p)
        return static_fail(PRAD_ERR_CUDA, "ledger_totals_noalloc: cudaGetSymbolAddress failed");
      if (cudaDeviceGetAttribute(&g_static_sms[dev], cudaDevAttrMultiProcessorCount, dev) !=
          cudaSuccess)
        return static_fail(PRAD_ERR_CUDA, "ledger_totals_noalloc: no multiprocessor count");
      g_static_addr[dev] = p;
    }
    scratch = g_static_addr[dev];
    sms = g_static_sms[dev];
  }
  if (n == 0) {  // nothing to read: zero totals without touching the inputs
    const cudaError_t ez = cudaMemsetAsync(out, 0, 2 * sizeof(double),
                                           static_cast<cudaStream_t>(stream));
    return ez == cudaSuccess ? PRAD_OK : static_fail(PRAD_ERR_CUDA, cudaGetErrorString(ez));
  }
  // the launch zeroes its scratch first: nothing left from an earlier call is
  // used
  const cudaError_t e = prad::launch_ledger_reduce(emit, rr, n, scratch, sms, out,
                                                   static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return static_fail(PRAD_ERR_CUDA, cudaGetErrorString(e));
  return PRAD_OK;
}
