// 16-bit-storage FFT: complex values stored in HBM as two FP16 or two BF16
// halves (4 bytes per point), transformed in FP32 in registers and shared
// memory (paper Sec. IX-A mixed-precision future work: half the bytes for
// SNR-limited radar data).  The passes are the single-CTA Stockham passes of
// stockham.cuh; only the first load (16-bit -> FP32, exact) and the last
// store (FP32 -> 16-bit, round to nearest; FP16 overflows to infinity, BF16
// keeps the FP32 range with 8 significant bits) differ.  The output is
// scaled (1/N for the inverse) before rounding.
//
// At half the bytes these launches are bound by the SM (shared-memory
// exchanges and arithmetic at about 60 % of their rates each), not by HBM.
// One tile per CTA: the plain kernel's tile loop needs 72 registers here (the
// raw 16-bit refill stays live beside the FP32 points) and measured slower
// (256 52.9 us against 45.5, 16384 124 against 91.6 us per 2^25 points).
// What it shares with the plain kernel measured, before / after: programmatic
// dependent launch, the twiddle read-ahead, the paired last pass, twiddle
// mode 1 at 4096 and the look-ahead prefetch 512 52.4 / 50.3, 1024 55.4 /
// 53.6, 2048 57.4 / 55.3, 4096 65.6 / 60.4, 8192 68.2 / 66.2, 16384 104.3 /
// 91.7 us.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "stockham.cuh"

namespace fftgb {

// The pair type's conversions: S2 = __half2 (FP16) or __nv_bfloat162 (BF16).
__device__ __forceinline__ float2 pair_to_float2(__half2 v) { return __half22float2(v); }
__device__ __forceinline__ float2 pair_to_float2(__nv_bfloat162 v) { return __bfloat1622float2(v); }
template <class S2>
__device__ __forceinline__ S2 float2_to_pair(float2 v);
template <>
__device__ __forceinline__ __half2 float2_to_pair<__half2>(float2 v) { return __float22half2_rn(v); }
template <>
__device__ __forceinline__ __nv_bfloat162 float2_to_pair<__nv_bfloat162>(float2 v) {
  return __float22bfloat162_rn(v);
}

template <class S2>
__device__ __forceinline__ void store_pairs(S2 *p, float2 u, float2 v) {  // two points, one access
  const S2 a = float2_to_pair<S2>(u), b = float2_to_pair<S2>(v);
  __stcs(reinterpret_cast<uint2 *>(p), make_uint2(*reinterpret_cast<const unsigned *>(&a),
                                                  *reinterpret_cast<const unsigned *>(&b)));
}

struct HalfArgs {
  const void *in;   // __half2 or __nv_bfloat162 pairs, per the kernel's S2
  void *out;
  const float2 *tw;
  long long batch;
  float scale;
  long long ahead;  // resident CTAs (the look-ahead prefetch); 0: none
};

template <int N, int P, int TB, int D, class SC, int TWM, class S2>
__global__ void __launch_bounds__(TB *(N / P))
stockham_half_kernel(HalfArgs args) {
  static_assert(SC::product() == N, "radix schedule must multiply to N");
  constexpr int T = N / P;
  constexpr bool PAIR_LAST = pairable<N, P, SC>();
  extern __shared__ __align__(128) float2 smem[];
  // Programmatic dependent launch, as the plain kernel.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int b = threadIdx.x / T;
  const int lt = threadIdx.x - b * T;
  float2 *buf = smem + b * N;
  const long long row = (long long)blockIdx.x * TB + b;
  const bool active = row < args.batch;
  if (args.ahead > 0 && threadIdx.x < 32) {
    const long long r2 = ((long long)blockIdx.x + args.ahead) * TB;
    if (r2 < args.batch) {
      const long long rows = args.batch - r2 < TB ? args.batch - r2 : TB;
      prefetch_l2_warp(static_cast<const S2 *>(args.in) + r2 * N, rows * N * (long long)sizeof(S2),
                       threadIdx.x);
    }
  }
  float2 a[P];
  const S2 *src = static_cast<const S2 *>(args.in) + row * N;
  if (active) {
#pragma unroll
    for (int m = 0; m < P; ++m) a[m] = pair_to_float2(__ldcs(src + lt + m * T));
  } else {
#pragma unroll
    for (int m = 0; m < P; ++m) a[m] = make_float2(0.f, 0.f);
  }
  run_passes_early<N, P, D, SC, 0, TWM, PAIR_LAST>(a, lt, buf, args.tw, NoHook{}, NoTw{});
  if (active) {
    S2 *dst = static_cast<S2 *>(args.out) + row * N;
    const float s = args.scale;
    if constexpr (PAIR_LAST) {
#pragma unroll
      for (int j = 0; j < P / 2; ++j)
        store_pairs(dst + final_index_pair<N, P, SC>(lt, j), cscale(a[2 * j], s),
                    cscale(a[2 * j + 1], s));
    } else {
#pragma unroll
      for (int m = 0; m < P; ++m)
        __stcs(dst + final_index<N, P, SC>(lt, m), float2_to_pair<S2>(cscale(a[m], s)));
    }
  }
}

}  // namespace fftgb
