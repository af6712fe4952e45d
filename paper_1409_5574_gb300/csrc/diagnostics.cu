// Angular distribution of the emitted energy (Fig. 4 of arXiv:1409.5574: the
// emitted energy over the front hemisphere around the laser propagation
// direction).  Each held photon record adds energy x weight to the bin of
// its direction: polar angle theta from the axis (bins uniform over
// [0, theta_max]) and azimuth phi around it, measured from the projection of
// a reference vector (bins uniform over [0, 2 pi)).  Block-private FP64
// histograms in shared memory, added to the output with one atomic per bin
// and block (FP64 sums: the order of the adds varies between runs in the
// last bits).
#include <cuda_runtime.h>
#include <stdint.h>

#include "prad_internal.h"

namespace prad {

namespace {

constexpr double kTwoPi = 6.283185307179586476925286766559;
constexpr int kUnsure = -2;  // (-1: beyond theta_max, or not a direction)

// The bin of a direction by the definition, in FP64.
__device__ __noinline__ int exact_bin(const AngularArgs& a, float fx, float fy, float fz) {
  const double nx = fx, ny = fy, nz = fz;
  const double c = nx * a.axis[0] + ny * a.axis[1] + nz * a.axis[2];
  const double th = acos(fmin(fmax(c, -1.0), 1.0));
  if (!(th <= a.theta_max)) return -1;  // also drops NaN directions
  const double p1 = nx * a.e1[0] + ny * a.e1[1] + nz * a.e1[2];
  const double p2 = nx * a.e2[0] + ny * a.e2[1] + nz * a.e2[2];
  double ph = atan2(p2, p1);
  if (ph < 0.0) ph += kTwoPi;
  int it = static_cast<int>(th * (a.ntheta / a.theta_max));
  int ip = static_cast<int>(ph * (a.nphi / kTwoPi));
  it = it < a.ntheta ? it : a.ntheta - 1;
  ip = ip < a.nphi ? (ip >= 0 ? ip : 0) : a.nphi - 1;
  return it * a.nphi + ip;
}

// The same from FP32 angles where these are sure of it.  The FP64 acos and
// atan2 of every record kept the FP64 pipe (2 lanes per clock and SM) busy for
// 1258 us on 6.3M records, 102 us so; only records closer to an edge than the
// FP32 error take them now.  Bounds of that error: the three products and
// sums of a component, of magnitude at most 1.0000002 with axes rounded to
// FP32, are off by at most 3e-7 = kDot; so theta, and acosf adds at most
// 4 ulp (1e-6): |dtheta| <= kDot / sin(theta) + 1e-6 while sin(theta) stays
// above 1e-2 (the second-order term is then below a hundredth of it) and at
// most sqrt(2 kDot) = 7.8e-4 closer to the axis, and |dphi| <= 2 kDot / rho +
// 2e-6 with rho the length across the axis.  Directions within 1e-5 of the axis
// are left to FP64, and the margins are doubled.  (The beam's own axis is where
// a good part of the records lie: with every direction within 1e-2 of it left
// to FP64 the kernel took 260 us.)
struct FastBins {
  float ax[3], e1[3], e2[3], per_t, per_p;
  int ntheta, nphi;
  __device__ explicit FastBins(const AngularArgs& a) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      ax[k] = static_cast<float>(a.axis[k]);
      e1[k] = static_cast<float>(a.e1[k]);
      e2[k] = static_cast<float>(a.e2[k]);
    }
    per_t = static_cast<float>(a.ntheta / a.theta_max);
    per_p = static_cast<float>(a.nphi / kTwoPi);
    ntheta = a.ntheta;
    nphi = a.nphi;
  }
  __device__ __forceinline__ int bin(float x, float y, float z) const {
    constexpr float kDot = 3e-7f;
    const float c = x * ax[0] + y * ax[1] + z * ax[2];
    const float p1 = x * e1[0] + y * e1[1] + z * e1[2];
    const float p2 = x * e2[0] + y * e2[1] + z * e2[2];
    const float rho2 = p1 * p1 + p2 * p2;
    // (a direction of another length than 1, or NaN, is left to FP64)
    if (!(rho2 > 1e-10f && fabsf(rho2 + c * c - 1.0f) < 1e-5f)) return kUnsure;
    const float inv = rsqrtf(rho2);
    // (c rounds beyond +-1 close to the axis or its opposite, and acosf is NaN
    // there: clamped as the definition does, which moves c no further off)
    const float t = acosf(fminf(fmaxf(c, -1.0f), 1.0f)) * per_t;
    float ph = atan2f(p2, p1);
    ph = (ph < 0.0f ? ph + static_cast<float>(kTwoPi) : ph) * per_p;
    const float dt = rho2 > 1e-4f ? kDot * inv : 7.8e-4f;
    const float mt = 2.0f * (dt + 1e-6f) * per_t + 2.4e-7f * t;
    const float mp = 2.0f * (2.0f * kDot * inv + 2e-6f) * per_p + 2.4e-7f * ph;
    // (written so that a NaN is unsure)
    if (!(fabsf(t - rintf(t)) > mt && fabsf(ph - rintf(ph)) > mp)) return kUnsure;
    const int it = static_cast<int>(t), ip = static_cast<int>(ph);
    if (it >= ntheta) return -1;
    return ip < nphi ? it * nphi + ip : kUnsure;
  }
};

// 512 threads share a block's bins, two blocks per SM: the adds are compare and
// swap loops on shared memory, whose latency wants warps to hide it, while
// every block more adds its bins to the output once more (256 x 2: 152 us, 512
// x 2: 102, 512 x 3: 128, 1024 x 1: 108 on 6.3M records).
constexpr int kHistThreads = 512, kHistBlocks = 2;
__global__ void __launch_bounds__(kHistThreads, kHistBlocks) k_angular_hist(AngularArgs a) {
  extern __shared__ double hist[];
  const int nb = a.ntheta * a.nphi;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) hist[b] = 0.0;
  __syncthreads();
  const unsigned long long cur = *a.cursor;
  const unsigned long long held =
      cur < static_cast<unsigned long long>(a.cap) ? cur : static_cast<unsigned long long>(a.cap);
  const FastBins f(a);
  for (unsigned long long i = blockIdx.x * static_cast<unsigned long long>(blockDim.x) + threadIdx.x;
       i < held; i += static_cast<unsigned long long>(gridDim.x) * blockDim.x) {
    const float fx = a.nx[i], fy = a.ny[i], fz = a.nz[i];
    const int bin = f.bin(fx, fy, fz);
    int at = bin;
    if (bin == kUnsure) at = exact_bin(a, fx, fy, fz);
    if (at < 0) continue;
    atomicAdd(&hist[at],
              static_cast<double>(a.eps[i]) * static_cast<double>(a.weight[i]));
  }
  __syncthreads();
  for (int b = threadIdx.x; b < nb; b += blockDim.x)
    if (hist[b] != 0.0) atomicAdd(a.out + b, hist[b]);
}

}  // namespace

cudaError_t launch_angular_hist(const AngularArgs& a, int num_sms, cudaStream_t s) {
  const size_t smem = sizeof(double) * static_cast<size_t>(a.ntheta) * a.nphi;
  cudaError_t e = cudaFuncSetAttribute(k_angular_hist,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(a.out, 0, smem, s);
  if (e != cudaSuccess) return e;
  k_angular_hist<<<kHistBlocks * num_sms, kHistThreads, smem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace prad
