// Calibration kernels: the throughput ceiling of the library's own modular
// arithmetic on this GPU, measured with every SM busy and no memory traffic. They
// give a measured denominator for the integer-bound kernels beside the one derived
// from unit counts and clocks.
//   KS_CAL_BUTTERFLY: the forward butterfly of the moduli below 2^51 (bfly_fwd_c), nothing
//                     between stages.
//   KS_CAL_MAC:       the exact multiply-accumulates of the basis conversions and the key
//                     multiply (Mac3), one reduction per 8 terms.
// (Before, with a conditional subtraction per butterfly and the 128-bit carry chain of the
// single-pass kernels, they read 0.905 T butterflies and 1.33 T terms a second, which the
// two-pass kernels exceed; now 1.126 T and 1.909 T on a GB300 at 2070 MHz.)
#include <cuda_runtime.h>

#include <algorithm>

#include "ks_arith.cuh"
#include "ks_internal.h"
#include "ks_ntt.cuh"

namespace ks {
namespace {

constexpr int kCalThreads = 256;
constexpr int kChains = 8;  // independent dependency chains per thread

__global__ void __launch_bounds__(kCalThreads) k_cal_butterfly(u64 m, u64 w, u64 wp, int iters,
                                                               u64 *sink) {
  u64 a[kChains], b[kChains];
#pragma unroll
  for (int c = 0; c < kChains; ++c) {
    a[c] = (threadIdx.x * 7919ull + c * 104729ull + blockIdx.x) % m;
    b[c] = (threadIdx.x * 15485863ull + c * 32452843ull) % m;
  }
  const ulonglong2 tw = make_ulonglong2(w, wp);
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int c = 0; c < kChains; ++c) bfly_fwd_c<CLS_FAST>(a[c], b[c], tw, m, 0);
  }
  u64 acc = 0;
#pragma unroll
  for (int c = 0; c < kChains; ++c) acc ^= a[c] ^ b[c];
  if (acc == 0x5eed) sink[blockIdx.x] = acc;  // practically never: defeats elimination
}

__global__ void __launch_bounds__(kCalThreads) k_cal_mac(u64 m, u64 minv, u64 c0, int iters,
                                                         u64 *sink) {
  u64 x[kChains], z[kChains];
#pragma unroll
  for (int c = 0; c < kChains; ++c) {
    x[c] = (threadIdx.x * 7919ull + c * 104729ull + blockIdx.x) % m;
    z[c] = 0;
  }
  const uint32_t inv = 0u - (uint32_t)minv;
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int c = 0; c < kChains; ++c) {
      Mac3 acc = {};
#pragma unroll
      for (int k = 0; k < 8; ++k) acc.add(x[c] + k, c0 + k);
      z[c] += acc.reduce(m, inv);
      x[c] = z[c] & ((1ull << 49) - 1);
    }
  }
  u64 acc = 0;
#pragma unroll
  for (int c = 0; c < kChains; ++c) acc ^= z[c];
  if (acc == 0x5eed) sink[blockIdx.x] = acc;
}

}  // namespace
}  // namespace ks

extern "C" int ks_calibrate(int kind, int iters, double *ops_per_s, void *stream) {
  using namespace ks;
  if (!ops_per_s || iters < 1 || (kind != KS_CAL_BUTTERFLY && kind != KS_CAL_MAC))
    return KS_EINVAL;
  int dev = 0, sms = 0, per_sm = 0;
  if (cudaGetDevice(&dev) || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) {
    cudaGetLastError();
    return KS_ECUDA;
  }
  cudaError_t e =
      kind == KS_CAL_BUTTERFLY
          ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_cal_butterfly, kCalThreads, 0)
          : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_cal_mac, kCalThreads, 0);
  if (e != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    return KS_ECUDA;
  }
  const int grid = sms * per_sm;
  cudaStream_t s = (cudaStream_t)stream;
  u64 *sink = nullptr;
  cudaEvent_t a = nullptr, b = nullptr;
  if (cudaMalloc(&sink, (size_t)grid * sizeof(u64)) || cudaEventCreate(&a) ||
      cudaEventCreate(&b)) {
    cudaGetLastError();
    if (sink) cudaFree(sink);
    if (a) cudaEventDestroy(a);
    return KS_ENOMEM;
  }
  // a 50-bit prime, a twiddle and its Shoup quotient floor(w 2^64 / m)
  const u64 m = 1125899906842177ull, w = 987654321987ull;
  const u64 wp = (u64)(((unsigned __int128)w << 64) / m);
  u64 minv = 1;  // -m^-1 mod 2^64 by Newton iteration
  for (int k = 0; k < 6; ++k) minv *= 2 - m * minv;
  minv = 0 - minv;
  auto launch = [&](int n) {
    if (kind == KS_CAL_BUTTERFLY)
      k_cal_butterfly<<<grid, kCalThreads, 0, s>>>(m, w, wp, n, sink);
    else
      k_cal_mac<<<grid, kCalThreads, 0, s>>>(m, minv, 0x123456789abull, n, sink);
  };
  launch(std::max(1, iters / 10));  // warm-up
  cudaEventRecord(a, s);
  launch(iters);
  cudaEventRecord(b, s);
  int rc = KS_OK;
  if (cudaEventSynchronize(b) != cudaSuccess) {
    rc = KS_ECUDA;
  } else {
    float ms = 0.f;
    cudaEventElapsedTime(&ms, a, b);
    const double per_iter = kind == KS_CAL_BUTTERFLY ? kChains : 8.0 * kChains;
    *ops_per_s = (double)grid * kCalThreads * iters * per_iter / (ms * 1e-3);
  }
  cudaGetLastError();
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  cudaFree(sink);
  return rc;
}
