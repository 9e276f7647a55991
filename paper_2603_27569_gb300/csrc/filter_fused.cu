// Fused spectral filter: y = IFFT(FFT(x) * H) in one kernel per row, its
// backward and its training step, for the SAR range-compression layer (paper
// Sec. II-D; the fused FFT -> matched filter -> IFFT pipeline is the paper's
// future work, Sec. IX-A).
//
//   forward   y = G (F x * H) (conj_h: * conj(H)), X_save = F x (optional)
//   backward  g_z = G^H g_y = F g_y / N; grad_H = sum_rows conj(X) * g_z;
//             grad_x = F^H (conj(H) * g_z)
//   step      both, for the loss L = sum m |y|^2, with g_y = 2 m y
//
// Every kernel keeps a row in registers from its load to its store: the
// transforms are those of specrow.cuh, whose spectrum stays in the order the
// forward leaves it in (pointwise work does not care) and whose time-domain
// side is in natural order, so a forward, a multiply and an inverse follow
// each other with no reordering between them.  All are persistent: CTA c
// takes tiles c, c + G, ... of TB rows (G = gridDim.x), refills each register
// with the next tile's point as it stores, and has warp 0 prefetch the tile
// after into L2.  Arrays that belong to a CTA for its whole life (H, the
// grad_H partial sums) or for a row (the step's X) live in tensor memory:
// each thread owns its lane and 2 P columns per array, the points of its P
// registers.  The grad_H sums run over a CTA's rows in row order, each CTA
// writes one partial row, and a fixed-order tree adds those: bitwise
// reproducible for a given grid.
//
// Bound by the SM, not by HBM: at 8192 the step runs its FMA pipe at 57 % and
// its L1 / shared-memory data pipe at 60 % with 14 warps per SM, DRAM at 40 %
// (ncu).  Per 2^25 points, us, with Stockham transforms that met in natural
// order (five exchanges per pair, generic accesses, twiddle rows through L1;
// three kernels for the backward below 8192) / now:
//            forward     + spectrum   backward     step
//     256    134 / 91    155 / 131    293 / 140    367 / 182
//    1024    174 / 101   196 / 133    288 / 141    481 / 221
//    4096    177 / 131   191 / 140    295 / 166    457 / 277
//    8192    162 / 134   181 / 146    212 / 175    359 / 297
//   16384    204 / 152   226 / 163    258 / 206    425 / 340
// (spectrum and backward in packed order; in natural order, for callers of
// the unpacked entry points, 130..193 and 146..244.)
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <new>

#include "plan.h"
#include "specrow.cuh"
#include "tmem.cuh"

namespace fftgb {

// Points moved between registers and tensor memory at a time.
template <int P>
constexpr int kChunk = P == 32 ? 8 : 4;
__device__ __forceinline__ void tmem_ld(uint32_t a, float (&r)[16]) { tmem_ld16(a, r); }
__device__ __forceinline__ void tmem_ld(uint32_t a, float (&r)[8]) { tmem_ld8(a, r); }
__device__ __forceinline__ void tmem_st(uint32_t a, const float (&r)[16]) { tmem_st16(a, r); }
__device__ __forceinline__ void tmem_st(uint32_t a, const float (&r)[8]) { tmem_st8(a, r); }

__device__ __forceinline__ float4 pack2(float2 a, float2 b) { return make_float4(a.x, a.y, b.x, b.y); }
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }

// Tensor-memory columns of one array (2 P per thread, every lane).
template <class R, int TB>
__host__ __device__ constexpr int array_cols() {
  return TB * R::T / 128 * 2 * R::P;
}
// Dynamic shared memory: TB row buffers, the twiddle rows, the address slot.
template <class R, int TB>
__host__ __device__ constexpr size_t filter_smem() {
  return sizeof(float2) * ((size_t)TB * R::BUF + R::TW + 2);
}
// CTAs per SM that registers are budgeted for: 128 per thread with 32 points;
// with 16 points 80 (three CTAs of 256 threads) or 64 (four), whichever measured
// faster (2^25 points, us, 80 / 64 registers, at 256, 512, 1024, 2048, 4096:
// forward 93 / 94, 96 / 110, 102 / 102, 112 / 109, 131 / 135; backward 141 /
// 157, 142 / 179, 142 / 170, 147 / 179, 169 / 168; step 182 / 198, 215 / 237,
// 221 / 248, 241 / 258, 293 / 277).  Spills by -Xptxas -v, bytes: forward none;
// backward 0 to 32 at 80 registers, 72 to 84 at 64, 40 to 48 at 128; step 0 to
// 36, 28, 120 to 152.
enum FilterKind { FK_FWD, FK_BWD, FK_STEP };
template <class R, int TB>
__host__ __device__ constexpr int filter_min_ctas(FilterKind k) {
  const int regs = R::P == 32 ? 128 : R::N == 4096 && k != FK_FWD ? 64 : 80;
  return 65536 / (TB * R::T * regs);
}

// Does the tensor-memory allocation stand before the first row's loads, or
// behind them, covered by their latency but with the row's registers held
// across it?  Measured, 2^25 points (1500 rows), us, before / behind: forward
// 256 93.3 / 93.1, 1024 101.2 / 102.4 (8.4 / 8.6), 8192 134.0 / 135.7, 16384
// 152.0 / 152.7; backward 256 150 / 141, 512 145.5 / 142.4 (11.1 / 11.4), 1024
// 141.5 / 142.2 (14.9 / 16.4), 2048 149.1 / 147.3 (23.0 / 22.3), 4096 166 / 167,
// 8192 175 / 176, 16384 210 / 206; step 1024 221 / 232, 2048 241 / 251, 4096
// 286 / 277, 8192 equal.
template <class R>
__host__ __device__ constexpr bool allocate_first(FilterKind k) {
  return k == FK_FWD   ? R::N >= 1024
         : k == FK_BWD ? R::N == 1024 || R::N == 4096 || R::N == 8192
                       : R::N <= 2048;
}

// What the filter kernels share: the CTA's tables and tensor memory, this
// thread's row slot, and the loads of its points.
template <class R, int TB, int NARRAYS>
struct FilterCta {
  static constexpr int N = R::N, P = R::P, T = R::T, NT = TB * T, WARPS = NT / 32;
  static_assert(NT % 128 == 0, "whole warpgroups cover the tensor-memory lanes");
  static constexpr uint32_t COLS = array_cols<R, TB>(), NCOL = COLS * NARRAYS;
  static_assert(NCOL >= 32 && NCOL <= 512 && (NCOL & (NCOL - 1)) == 0, "allocatable");
  int tid, warp, b, lt;
  float2 *buf, *tw;
  uint32_t tbase, taddr;

  // Before the dependency wait: the tables are constant from the plan's
  // creation on.
  __device__ __forceinline__ FilterCta(float2 *smem, const float2 *tables) {
    tid = threadIdx.x;
    warp = tid >> 5;
    b = tid / T;
    lt = tid - b * T;
    buf = smem + b * R::BUF;
    tw = smem + TB * R::BUF;
    R::Rows::copy(tw, tables, tid, NT);
  }
  // After the wait (tmem.cuh): warp 0 allocates, and the barrier publishes the
  // address and the tables (and H, where it is staged).
  __device__ __forceinline__ uint32_t *slot() const { return reinterpret_cast<uint32_t *>(tw + R::TW); }
  __device__ __forceinline__ void allocate() const {
    if (warp == 0) tmem_alloc_warp(slot(), NCOL);
  }
  __device__ __forceinline__ void publish() {
    tmem_fence_before();
    __syncthreads();
    tmem_fence_after();
    tbase = *slot();
    taddr = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(2 * P * (warp >> 2));
  }
  __device__ __forceinline__ uint32_t array(int i) const { return taddr + COLS * i; }
  __device__ __forceinline__ void release() const {
    tmem_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc_warp(tbase, NCOL);
  }
  static __device__ __forceinline__ void load(float2 (&v)[P], const float2 *row, int lt, bool on) {
#pragma unroll
    for (int m = 0; m < P; ++m) v[m] = on ? __ldcs(row + lt + m * T) : make_float2(0.f, 0.f);
  }
  __device__ __forceinline__ void prefetch(const void *base, long long tile, long long batch,
                                           int point_bytes) const {
    if (warp == 0) {
      const long long rows = batch - tile * TB < TB ? batch - tile * TB : TB;
      prefetch_l2_warp(static_cast<const char *>(base) + tile * TB * N * point_bytes,
                       rows * N * point_bytes, tid);
    }
  }
  __device__ __forceinline__ void zero(uint32_t t) const {
    float z[2 * kChunk<P>];
#pragma unroll
    for (int i = 0; i < 2 * kChunk<P>; ++i) z[i] = 0.f;
#pragma unroll
    for (int c = 0; c < P / kChunk<P>; ++c) tmem_st(t + 2 * kChunk<P> * c, z);
    tmem_wait_st();
  }
  // Place of natural-order entry k in the row buffer: reads and writes by
  // frequency meet 2-way bank conflicts instead of 8-way.
  static __device__ __forceinline__ constexpr int at(int k) { return k + 2 * (k >> 5); }
  static_assert(at(N - 1) < R::BUF, "a natural-order row fits the buffer");

  // H (or conj(H)) at this thread's frequencies into the array at t, once.
  // Rows that fill a CTA get it through the row buffer: read in order, in
  // flight beside the row's own loads (issued between the two calls).  Gathers
  // from global memory touch 16 lines per warp load there and wait for each
  // chunk.  Below, gathers touch fewer lines and are shared by the CTA's rows.
  // Forward of one row / 400 rows / 2^25 points, us, gathered / staged: 1024
  // 3.6 / 3.9, 3.9 / 4.4, 102 / 103; 4096 4.9 / 4.6, 11.5 / 9.7, 132 / 131;
  // 8192 8.4 / 7.7, 22.3 / 19.9, 135 / 134; 16384 15.2 / 13.9, 38.2 / 36.5,
  // 154 / 153.
  static constexpr bool STAGE_H = TB == 1;
  __device__ __forceinline__ void fetch_h(const float2 *H) const {
    if constexpr (STAGE_H) {
      const uint32_t to = (uint32_t)__cvta_generic_to_shared(buf);
#pragma unroll
      for (int m = 0; m < P; ++m) {
        const int k = lt + m * T;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(to + 8 * at(k)), "l"(H + k)
                     : "memory");
      }
    }
  }
  __device__ __forceinline__ void land_h() const {  // publish() follows
    if constexpr (STAGE_H) asm volatile("cp.async.wait_all;" ::: "memory");
  }
  __device__ __forceinline__ void stash_h(const R &r, const float2 *H, bool conj, uint32_t t) const {
    constexpr int C = kChunk<P>;
#pragma unroll
    for (int c = 0; c < P / C; ++c) {
      float h[2 * C];
#pragma unroll
      for (int q = 0; q < C; ++q) {
        const int k = r.freq(C * c + q);
        const float2 w = STAGE_H ? buf[at(k)] : __ldg(H + k);
        h[2 * q] = w.x;
        h[2 * q + 1] = conj ? -w.y : w.y;
      }
      tmem_st(t + 2 * C * c, h);
    }
    if constexpr (STAGE_H) R::template row_sync<TB>(b);  // the buffer is the transforms' again
    tmem_wait_st();
  }
  // v *= the array at t
  static __device__ __forceinline__ void multiply(float2 (&v)[P], uint32_t t) {
    constexpr int C = kChunk<P>;
#pragma unroll
    for (int c = 0; c < P / C; ++c) {
      float h[2 * C];
      tmem_ld(t + 2 * C * c, h);
      tmem_wait_ld(h);
#pragma unroll
      for (int q = 0; q < C; ++q)
        v[C * c + q] = cmul(v[C * c + q], make_float2(h[2 * q], h[2 * q + 1]));
    }
  }
  // sum += conj(x) g_z for one point
  static __device__ __forceinline__ void accumulate(float *s, float2 x, float2 g) {
    s[0] = fmaf(x.x, g.x, fmaf(x.y, g.y, s[0]));
    s[1] = fmaf(x.x, g.y, fmaf(-x.y, g.x, s[1]));
  }
  // The CTA's sums (array at t) as one packed row: its TB row slots added in
  // slot order through the row buffers.
  __device__ __forceinline__ void write_sums(uint32_t t, float2 *smem, float2 *dst) const {
    constexpr int C = kChunk<P>;
    __syncthreads();  // the buffers' last use is over
#pragma unroll
    for (int c = 0; c < P / C; ++c) {
      float s[2 * C];
      tmem_ld(t + 2 * C * c, s);
      tmem_wait_ld(s);
#pragma unroll
      for (int q = 0; q < C; q += 2) {
        const int pos = ((C * c + q) / 2 * T + lt) * 2;
        const float4 w = make_float4(s[2 * q], s[2 * q + 1], s[2 * q + 2], s[2 * q + 3]);
        *reinterpret_cast<float4 *>(TB == 1 ? dst + pos : smem + b * N + pos) = w;
      }
    }
    if constexpr (TB > 1) {
      __syncthreads();
      for (int k = tid; k < N; k += NT) {
        float2 acc = smem[k];
        for (int i = 1; i < TB; ++i) acc = cadd(acc, smem[i * N + k]);
        dst[k] = acc;
      }
    }
  }
};

struct FilterArgs {
  const float2 *in;       // x, or g_y
  float2 *out;            // y, or grad_x (may equal in)
  const float2 *H;        // [N]
  float2 *x_save;         // forward: F x (nullable); backward: the saved spectrum
  float2 *partial;        // backward: [gridDim.x][N] per-CTA grad_H sums, packed order
  const float2 *tw;
  long long batch;
  int conj_h;             // forward: multiply by conj(H) instead of H
  float inv_n;
};

// NATURAL: the saved spectrum leaves in natural order.  With two butterflies
// per thread (8192) registers m and m + P / 2 are adjacent frequencies and two
// lanes fill a sector, so the pairs are stored as they are.  The other lengths
// hold single points there and stage through the row buffer (an exchange and
// three row barriers more than the packed order).  Staged / stored directly,
// one row and 2^25 points, us: 8192 9.2 / 8.7 and 169 / 161; 4096 5.4 / 5.7 and
// 161 / 185; 16384 16.5 / 17.3 and 195 / 210.
template <class R, int TB, bool NATURAL>
__global__ void __launch_bounds__(TB *R::T, filter_min_ctas<R, TB>(FK_FWD))
filter_fwd_kernel(FilterArgs a) {
  constexpr int N = R::N, P = R::P, T = R::T;
  extern __shared__ __align__(128) float2 smem[];
  FilterCta<R, TB, 1> cta(smem, a.tw);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const R r(cta.buf, cta.lt, cta.b);
  const int lt = cta.lt;
  const long long ntiles = (a.batch + TB - 1) / TB;
  long long tile = blockIdx.x;
  if constexpr (allocate_first<R>(FK_FWD)) cta.allocate();
  cta.fetch_h(a.H);
  float2 v[P];
  {
    const long long row = tile * TB + cta.b;
    const bool on = row < a.batch;
    cta.load(v, a.in + (on ? row : 0) * N, lt, on);
  }
  if constexpr (!allocate_first<R>(FK_FWD)) cta.allocate();
  cta.land_h();
  cta.publish();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  cta.stash_h(r, a.H, a.conj_h, cta.array(0));
  for (; tile < ntiles; tile += gridDim.x) {
    const long long next = tile + gridDim.x;
    if (next < ntiles) cta.prefetch(a.in, next, a.batch, sizeof(float2));
    const long long row = tile * TB + cta.b, nrow = next * TB + cta.b;
    const bool active = row < a.batch, load_next = nrow < a.batch;
    r.template forward<TB>(v, cta.tw);
    if (a.x_save) {
      float2 *xs = a.x_save + (active ? row : 0) * N;
      if constexpr (NATURAL && R::QB == 2) {
        if (active) {
#pragma unroll
          for (int m = 0; m < P / 2; ++m)
            __stcs(reinterpret_cast<float4 *>(xs + r.freq(m)), pack2(v[m], v[m + P / 2]));
        }
      } else if constexpr (NATURAL) {
        R::template row_sync<TB>(cta.b);  // every sub-row has been read
#pragma unroll
        for (int m = 0; m < P; ++m) cta.buf[cta.at(r.freq(m))] = v[m];
        R::template row_sync<TB>(cta.b);
#pragma unroll
        for (int m = 0; m < P; ++m)
          if (active) __stcs(xs + lt + m * T, cta.buf[cta.at(lt + m * T)]);
        R::template row_sync<TB>(cta.b);
      } else if (active) {
#pragma unroll
        for (int m = 0; m < P; m += 2)
          __stcs(reinterpret_cast<float4 *>(xs + (m / 2 * T + lt) * 2), pack2(v[m], v[m + 1]));
      }
    }
    cta.multiply(v, cta.array(0));
    r.template inverse<TB>(v, cta.tw);
    float2 *dst = a.out + (active ? row : 0) * N + lt;
    const float2 *src = a.in + (load_next ? nrow : 0) * N + lt;
#pragma unroll
    for (int m = 0; m < P; ++m) {
      if (active) __stcs(dst + m * T, cscale(v[m], a.inv_n));
      if (load_next) v[m] = __ldcs(src + m * T);
    }
  }
  cta.release();
}

// PACKED: the saved spectrum is in packed order (coalesced 16-byte loads),
// else in natural order.
template <class R, int TB, bool PACKED>
__global__ void __launch_bounds__(TB *R::T, filter_min_ctas<R, TB>(FK_BWD))
filter_bwd_kernel(FilterArgs a) {
  constexpr int N = R::N, P = R::P, T = R::T, C = kChunk<P>;
  extern __shared__ __align__(128) float2 smem[];
  FilterCta<R, TB, 2> cta(smem, a.tw);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const R r(cta.buf, cta.lt, cta.b);
  const int lt = cta.lt;
  const long long ntiles = (a.batch + TB - 1) / TB;
  long long tile = blockIdx.x;
  if constexpr (allocate_first<R>(FK_BWD)) cta.allocate();
  cta.fetch_h(a.H);
  float2 v[P];
  {
    const long long row = tile * TB + cta.b;
    const bool on = row < a.batch;
    cta.load(v, a.in + (on ? row : 0) * N, lt, on);
  }
  cta.prefetch(a.x_save, tile, a.batch, sizeof(float2));
  if constexpr (!allocate_first<R>(FK_BWD)) cta.allocate();
  cta.land_h();
  cta.publish();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t t_sum = cta.array(0), t_h = cta.array(1);
  cta.stash_h(r, a.H, true, t_h);
  cta.zero(t_sum);
  for (; tile < ntiles; tile += gridDim.x) {
    const long long next = tile + gridDim.x;
    if (next < ntiles) {
      cta.prefetch(a.in, next, a.batch, sizeof(float2));
      cta.prefetch(a.x_save, next, a.batch, sizeof(float2));
    }
    const long long row = tile * TB + cta.b, nrow = next * TB + cta.b;
    const bool active = row < a.batch, load_next = nrow < a.batch;
    const bool on = TB == 1 || active;  // a row past the batch adds zeros
    const float2 *xs = a.x_save + (active ? row : 0) * N;
    r.template forward<TB>(v, cta.tw);
#pragma unroll
    for (int m = 0; m < P; ++m) v[m] = cscale(v[m], a.inv_n);  // g_z
    // The spectrum is read one chunk ahead of the sums it goes into.
    float2 x[2][C];
    auto load_x = [&](int c) {
#pragma unroll
      for (int q = 0; q < C; q += 2) {
        const int m = C * c + q;
        float2 *to = x[c & 1] + q;
        if constexpr (PACKED) {
          const float4 w = on ? __ldcs(reinterpret_cast<const float4 *>(xs + (m / 2 * T + lt) * 2))
                              : make_float4(0.f, 0.f, 0.f, 0.f);
          to[0] = lo2(w);
          to[1] = hi2(w);
        } else {
          to[0] = on ? xs[r.freq(m)] : make_float2(0.f, 0.f);
          to[1] = on ? xs[r.freq(m + 1)] : make_float2(0.f, 0.f);
        }
      }
    };
    load_x(0);
#pragma unroll
    for (int c = 0; c < P / C; ++c) {
      float s[2 * C];
      tmem_ld(t_sum + 2 * C * c, s);
      if (c + 1 < P / C) load_x(c + 1);
      tmem_wait_ld(s);
#pragma unroll
      for (int q = 0; q < C; ++q) cta.accumulate(s + 2 * q, x[c & 1][q], v[C * c + q]);
      tmem_st(t_sum + 2 * C * c, s);
    }
    cta.multiply(v, t_h);
    tmem_wait_st();
    r.template inverse<TB>(v, cta.tw);
    float2 *dst = a.out + (active ? row : 0) * N + lt;
    const float2 *src = a.in + (load_next ? nrow : 0) * N + lt;
#pragma unroll
    for (int m = 0; m < P; ++m) {
      if (active) __stcs(dst + m * T, v[m]);
      v[m] = load_next ? __ldcs(src + m * T) : make_float2(0.f, 0.f);
    }
  }
  cta.write_sums(t_sum, smem, a.partial + (size_t)blockIdx.x * N);
  cta.release();
}

// Fused training step for the masked-energy loss L = sum m |y|^2 (m real, one
// value per point).  Per row: X = F x (kept in tensor memory); y = G (X H),
// stored; L += m |y|^2; g_y = 2 m y; g_z = F g_y / N; sums += conj(X) g_z;
// grad_x = F^H (conj(H) g_z).  X and g_y never leave the SM: a row reads x
// and m and writes y and grad_x, 28 bytes per point.  Tensor memory holds the
// sums and X, so H comes from a copy in packed order that a small kernel
// before this one leaves in grad_H (coalesced 16-byte loads): the caller's
// buffer, which nothing else uses before the tree writes the result there, so
// that steps of one plan on two streams read each its own H.
struct FilterStepArgs {
  const float2 *x;
  const float2 *hp;   // H, packed order
  const float *mask;  // m, [batch][N]
  float2 *y;          // nullable
  float2 *gx;         // grad_x
  float2 *partial;    // [gridDim.x][N] per-CTA grad_H sums, packed order
  float *loss_part;   // [gridDim.x] per-CTA loss sums
  const float2 *tw;
  long long batch;
  float inv_n;
};

__global__ void pack_h_kernel(const float2 *H, float2 *hp, int N, SpecShape s) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) hp[i] = H[spec_freq(s, i)];
}

template <class R, int TB>
__global__ void __launch_bounds__(TB *R::T, filter_min_ctas<R, TB>(FK_STEP))
filter_step_kernel(FilterStepArgs a) {
  constexpr int N = R::N, P = R::P, T = R::T, C = kChunk<P>;
  constexpr int MK = P == 32 ? 16 : 2;  // registers allow 16 beside 32 points, not beside 16
  extern __shared__ __align__(128) float2 smem[];
  FilterCta<R, TB, 2> cta(smem, a.tw);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if constexpr (allocate_first<R>(FK_STEP)) cta.allocate();
  const R r(cta.buf, cta.lt, cta.b);
  const int lt = cta.lt;
  const long long ntiles = (a.batch + TB - 1) / TB;
  long long tile = blockIdx.x;
  float2 v[P];
  {
    const long long row = tile * TB + cta.b;
    const bool on = row < a.batch;
    cta.load(v, a.x + (on ? row : 0) * N, lt, on);
  }
  if constexpr (!allocate_first<R>(FK_STEP)) cta.allocate();
  cta.publish();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const uint32_t t_sum = cta.array(0), t_x = cta.array(1);
  cta.zero(t_sum);
  float loss = 0.f;
  for (; tile < ntiles; tile += gridDim.x) {
    const long long next = tile + gridDim.x;
    if (next < ntiles) {
      cta.prefetch(a.x, next, a.batch, sizeof(float2));
      cta.prefetch(a.mask, next, a.batch, sizeof(float));
    }
    const long long row = tile * TB + cta.b, nrow = next * TB + cta.b;
    const bool active = row < a.batch, load_next = nrow < a.batch;
    const long long r0 = active ? row : 0;  // a row past the batch holds zeros, stores nothing
    // The two halves share one body: the transforms' code exists once.
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      r.template forward<TB>(v, cta.tw);
      const float4 *hp = reinterpret_cast<const float4 *>(a.hp) + lt;
      if (half == 0) {
#pragma unroll
        for (int c = 0; c < P / C; ++c) {
          float x[2 * C];
#pragma unroll
          for (int q = 0; q < C; ++q) {
            x[2 * q] = v[C * c + q].x;
            x[2 * q + 1] = v[C * c + q].y;
          }
          tmem_st(t_x + 2 * C * c, x);
        }
#pragma unroll
        for (int m = 0; m < P; m += 2) {
          const float4 h = __ldg(hp + m / 2 * T);
          v[m] = cmul(v[m], lo2(h));
          v[m + 1] = cmul(v[m + 1], hi2(h));
        }
      } else {
#pragma unroll
        for (int c = 0; c < P / C; ++c) {
          float s[2 * C], x[2 * C];
          tmem_ld(t_sum + 2 * C * c, s);
          tmem_ld(t_x + 2 * C * c, x);
          tmem_wait_ld(s);
          tmem_wait_ld(x);
#pragma unroll
          for (int q = 0; q < C; q += 2) {
            const int m = C * c + q;
            const float4 h = __ldg(hp + m / 2 * T);
            const float2 g0 = cscale(v[m], a.inv_n), g1 = cscale(v[m + 1], a.inv_n);  // g_z
            cta.accumulate(s + 2 * q, make_float2(x[2 * q], x[2 * q + 1]), g0);
            cta.accumulate(s + 2 * q + 2, make_float2(x[2 * q + 2], x[2 * q + 3]), g1);
            v[m] = cmulc(g0, lo2(h));
            v[m + 1] = cmulc(g1, hi2(h));
          }
          tmem_st(t_sum + 2 * C * c, s);
        }
      }
      tmem_wait_st();
      r.template inverse<TB>(v, cta.tw);
      if (half == 0) {
        float2 *y = a.y ? a.y + r0 * N + lt : nullptr;
        const float *mk = a.mask + r0 * N + lt;
#pragma unroll
        for (int m0 = 0; m0 < P; m0 += MK) {  // MK mask loads in flight before the stores
          float w[MK];
#pragma unroll
          for (int i = 0; i < MK; ++i) w[i] = active ? __ldcs(mk + (m0 + i) * T) : 0.f;
#pragma unroll
          for (int i = 0; i < MK; ++i) {
            const int m = m0 + i;
            const float2 yv = cscale(v[m], a.inv_n);
            if (active && y) __stcs(y + m * T, yv);
            loss = fmaf(w[i], fmaf(yv.x, yv.x, yv.y * yv.y), loss);
            v[m] = cscale(yv, 2.f * w[i]);
          }
        }
      } else {
        float2 *dst = a.gx + r0 * N + lt;
        const float2 *src = a.x + (load_next ? nrow : 0) * N + lt;
#pragma unroll
        for (int m = 0; m < P; ++m) {
          if (active) __stcs(dst + m * T, v[m]);
          v[m] = load_next ? __ldcs(src + m * T) : make_float2(0.f, 0.f);
        }
      }
    }
  }
  cta.write_sums(t_sum, smem, a.partial + (size_t)blockIdx.x * N);
  // the CTA's loss: a fixed-order tree over the threads
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
  __syncthreads();  // the slot sums are read: the buffer takes the loss
  float *red = reinterpret_cast<float *>(smem);
  if ((cta.tid & 31) == 0) red[cta.warp] = loss;
  __syncthreads();
  if (cta.tid == 0) {
    float t = 0.f;
    for (int w = 0; w < cta.WARPS; ++w) t += red[w];
    a.loss_part[blockIdx.x] = t;
  }
  cta.release();
}

struct FilterKernel {
  const void *fn;
  int cols;  // tensor-memory columns per CTA
};

// The kernels of one N: 32 points per thread from 8192 on, 16 below; TB rows
// per CTA of 256 threads (512 at 16384).
struct FilterVariant {
  FilterKernel fwd, fwd_natural, bwd, bwd_natural, step;
  int threads, tb;
  size_t smem;
  SpecShape shape;
  KernelEntry sched;  // the schedule whose pass tables the transforms read
};

template <int N, int P, int TB, int RA>
static FilterVariant variant() {
  using R = SpecRow<N, P, RA>;
  constexpr int cols = array_cols<R, TB>();
  FilterVariant v;
  v.fwd = {(const void *)&filter_fwd_kernel<R, TB, false>, cols};
  v.fwd_natural = {(const void *)&filter_fwd_kernel<R, TB, true>, cols};
  v.bwd = {(const void *)&filter_bwd_kernel<R, TB, true>, 2 * cols};
  v.bwd_natural = {(const void *)&filter_bwd_kernel<R, TB, false>, 2 * cols};
  v.step = {(const void *)&filter_step_kernel<R, TB>, 2 * cols};
  v.threads = TB * R::T;
  v.tb = TB;
  v.smem = filter_smem<R, TB>();
  v.shape = R::shape();
  v.sched = KernelEntry{};
  v.sched.npass = R::Tables::npass;
  for (int i = 0; i < R::Tables::npass; ++i) v.sched.radix[i] = R::Tables::radix[i];
  return v;
}

static bool filter_variant(int N, FilterVariant *v) {
  switch (N) {
    case 256: *v = variant<256, 16, 16, 1>(); return true;
    case 512: *v = variant<512, 16, 8, 2>(); return true;
    case 1024: *v = variant<1024, 16, 4, 4>(); return true;
    case 2048: *v = variant<2048, 16, 2, 8>(); return true;
    case 4096: *v = variant<4096, 16, 1, 16>(); return true;
    case 8192: *v = variant<8192, 32, 1, 16>(); return true;
    case 16384: *v = variant<16384, 32, 1, 16>(); return true;
  }
  return false;
}

struct FilterState {
  FilterVariant v;
  float2 *d_work = nullptr;      // grad_H sums, one row per CTA and launch
  float2 *d_hp = nullptr;        // the training step's packed H, where grad_H cannot hold it
  float *d_loss_part = nullptr;  // per-CTA loss sums of the training step
  int fwd_grid = 0, bwd_grid = 0, step_grid = 0;
};

void filter_destroy(fft_plan_impl *pl) {
  FilterState *f = (FilterState *)pl->filter;
  if (f) {
    cudaFree(f->d_work);
    cudaFree(f->d_hp);
    cudaFree(f->d_loss_part);
  }
  delete f;
  pl->filter = nullptr;
}

// The backward below 8192 points runs in launches of at most kSumRows rows per
// row slot, each with its own rows of sums, so that no FP32 sum runs over more
// than kSumRows rows in order however large the batch; the pairwise tree adds
// them all.  (2^25 points are 18 rows per slot at most: one launch.)  From 8192
// points on the one launch's CTAs, two per SM or one, add their rows in order.
constexpr int kSumRows = 32;
struct BwdLaunches {
  int64_t rows;  // of each launch but the last
  int64_t sums;  // rows of sums of all
};
static BwdLaunches bwd_launches(const FilterVariant &v, int N, int64_t batch, int grid) {
  const int64_t round = (int64_t)grid * v.tb;
  if (N >= 8192 || batch <= kSumRows * round) return {batch, grid};
  const int64_t rows = kSumRows * round, full = (batch - 1) / rows;
  const int64_t rest = (batch - full * rows + v.tb - 1) / v.tb;
  return {rows, full * grid + std::min<int64_t>(grid, rest)};
}

// CTAs of kernel k that are resident on the GPU at once.  The occupancy query
// reports one per SM for any kernel that allocates tensor memory, while the
// hardware co-schedules as many as registers, shared memory and tensor memory
// allow (measured at 8192: two, 213 us against 270 us for the backward).
static int resident(const FilterKernel &k, const FilterVariant &v, int dev) {
  int sms = 0, smem_sm = 0, regs_sm = 0, reserved = 0, threads_sm = 0;
  cudaFuncAttributes at;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) !=
          cudaSuccess ||
      cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) !=
          cudaSuccess ||
      cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev) !=
          cudaSuccess ||
      cudaDeviceGetAttribute(&threads_sm, cudaDevAttrMaxThreadsPerMultiProcessor, dev) !=
          cudaSuccess ||
      cudaFuncGetAttributes(&at, k.fn) != cudaSuccess)
    return 0;
  const int regs = (at.numRegs + 7) / 8 * 8 * v.threads;
  const int by_smem = smem_sm / ((int)v.smem + (int)at.sharedSizeBytes + reserved);
  return sms * std::max(1, std::min({regs_sm / regs, by_smem, threads_sm / v.threads, 512 / k.cols}));
}

}  // namespace fftgb

using namespace fftgb;

extern "C" {

fft_status_t fft_filter_plan(fft_plan_t *out, int N, int64_t batch) {
  if (!out) return FFT_ERR_INVALID_VALUE;
  *out = nullptr;
  if (batch < 0 || N < 2 || N > 16384 || (N & (N - 1))) return FFT_ERR_INVALID_SIZE;
  FilterVariant v;
  if (!filter_variant(N, &v)) return FFT_ERR_NOT_SUPPORTED;
  fft_plan_s *h = new (std::nothrow) fft_plan_s;
  FilterState *f = new (std::nothrow) FilterState;
  if (!h || !f) {
    delete h;
    delete f;
    return FFT_ERR_ALLOC;
  }
  fft_plan_impl *pl = &h->impl;
  pl->N = N;
  pl->batch = batch;
  pl->path = FFT_PATH_FILTER;
  pl->filter = f;
  f->v = v;
  cudaGetDevice(&pl->device);
  auto fail = [&](fft_status_t e) {
    filter_destroy(pl);
    if (pl->d_tw) cudaFree(pl->d_tw);
    if (pl->d_status) cudaFree(pl->d_status);
    delete h;
    return e;
  };
  auto alloc = [](auto **p, int64_t bytes) {
    if (bytes <= 0 || dev_malloc(p, (size_t)bytes) == cudaSuccess) return true;
    cudaGetLastError();
    return false;
  };
  if (!alloc(&pl->d_status, sizeof(int))) return fail(FFT_ERR_ALLOC);
  cudaMemset(pl->d_status, 0, sizeof(int));
  for (const FilterKernel *k : {&v.fwd, &v.fwd_natural, &v.bwd, &v.bwd_natural, &v.step}) {
    if (v.smem > 48 * 1024 &&
        cudaFuncSetAttribute(k->fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)v.smem) !=
            cudaSuccess)
      return fail(FFT_ERR_CUDA);
  }
  int64_t off = 0;
  fft_status_t s = build_twiddles(pl, pass_segments(v.sched, off));
  if (s != FFT_OK) return fail(s);
  if (batch > 0) {
    const int64_t ntiles = (batch + v.tb - 1) / v.tb;
    auto grid = [&](const FilterKernel &k) {
      return (int)std::min<int64_t>(resident(k, v, pl->device), ntiles);
    };
    f->fwd_grid = grid(v.fwd);
    f->bwd_grid = grid(v.bwd);
    f->step_grid = grid(v.step);
    if (f->fwd_grid < 1 || f->bwd_grid < 1 || f->step_grid < 1) return fail(FFT_ERR_CUDA);
    const int64_t row = (int64_t)sizeof(float2) * N;
    pl->scratch_bytes =
        std::max<int64_t>(bwd_launches(v, N, batch, f->bwd_grid).sums, f->step_grid) * row;
    if (!alloc(&f->d_work, pl->scratch_bytes) || !alloc(&f->d_hp, row) ||
        !alloc(&f->d_loss_part, (int64_t)sizeof(float) * f->step_grid))
      return fail(FFT_ERR_ALLOC);
  }
  *out = h;
  return FFT_OK;
}

static fft_status_t filter_check(fft_plan_t plan, const void *a, const void *b, const void *c) {
  if (!plan || plan->impl.path != FFT_PATH_FILTER) return FFT_ERR_INVALID_VALUE;
  if (!a || !b || !c) return FFT_ERR_INVALID_VALUE;
  if (((uintptr_t)a | (uintptr_t)b | (uintptr_t)c) & 15) return FFT_ERR_MISALIGNED;
  return FFT_OK;
}

static bool overlap(const void *p, int64_t pb, const void *q, int64_t qb) {
  const char *a = (const char *)p, *b = (const char *)q;
  return a < b + qb && b < a + pb;
}

static fft_status_t filter_forward(fft_plan_t plan, const void *x, const void *H, void *y,
                                   void *X_save, int conj_h, bool natural, void *stream) {
  fft_status_t s = filter_check(plan, x, H, y);
  if (s != FFT_OK) return s;
  if ((uintptr_t)X_save & 15) return FFT_ERR_MISALIGNED;
  fft_plan_impl *pl = &plan->impl;
  FilterState *f = (FilterState *)pl->filter;
  if (pl->batch == 0) return FFT_OK;
  FilterArgs a{};
  a.in = (const float2 *)x;
  a.out = (float2 *)y;
  a.H = (const float2 *)H;
  a.x_save = (float2 *)X_save;
  a.tw = pl->d_tw;
  a.batch = pl->batch;
  a.conj_h = conj_h ? 1 : 0;
  a.inv_n = 1.0f / (float)pl->N;
  const int64_t bytes = (int64_t)sizeof(float2) * pl->N * pl->batch;
  // the saved spectrum may not overlap x or y (header contract)
  if (X_save && (overlap(X_save, bytes, x, bytes) || overlap(X_save, bytes, y, bytes)))
    return FFT_ERR_INVALID_VALUE;
  const FilterKernel &k = X_save && natural ? f->v.fwd_natural : f->v.fwd;
  void *args[] = {&a};
  return cuda_status(launch_pdl(k.fn, dim3((unsigned)f->fwd_grid), dim3(f->v.threads), f->v.smem,
                                (cudaStream_t)stream, args));
}

static fft_status_t filter_backward(fft_plan_t plan, const void *g_y, const void *H,
                                    const void *X_saved, void *grad_x, void *grad_H, bool natural,
                                    void *stream) {
  fft_status_t s = filter_check(plan, g_y, H, grad_x);
  if (s != FFT_OK) return s;
  if (!X_saved || !grad_H) return FFT_ERR_INVALID_VALUE;
  if (((uintptr_t)X_saved | (uintptr_t)grad_H) & 15) return FFT_ERR_MISALIGNED;
  fft_plan_impl *pl = &plan->impl;
  FilterState *f = (FilterState *)pl->filter;
  cudaStream_t st = (cudaStream_t)stream;
  const int N = pl->N;
  if (pl->batch == 0) return cuda_status(cudaMemsetAsync(grad_H, 0, sizeof(float2) * N, st));
  const int64_t bytes = (int64_t)sizeof(float2) * N * pl->batch;
  // grad_x may not overlap g_y or X_saved (header contract)
  if (overlap(grad_x, bytes, g_y, bytes) || overlap(grad_x, bytes, X_saved, bytes))
    return FFT_ERR_INVALID_VALUE;
  FilterArgs b{};
  b.in = (const float2 *)g_y;
  b.x_save = (float2 *)const_cast<void *>(X_saved);
  b.H = (const float2 *)H;
  b.out = (float2 *)grad_x;
  b.partial = f->d_work;
  b.tw = pl->d_tw;
  b.inv_n = 1.0f / (float)N;
  const FilterKernel &k = natural ? f->v.bwd_natural : f->v.bwd;
  const BwdLaunches l = bwd_launches(f->v, N, pl->batch, f->bwd_grid);
  for (int64_t r0 = 0; r0 < pl->batch; r0 += l.rows) {
    b.batch = std::min(l.rows, pl->batch - r0);
    const int64_t grid = std::min<int64_t>(f->bwd_grid, (b.batch + f->v.tb - 1) / f->v.tb);
    void *args[] = {&b};
    if ((s = cuda_status(launch_pdl(k.fn, dim3((unsigned)grid), dim3(f->v.threads), f->v.smem, st,
                                    args))) != FFT_OK)
      return s;
    b.in += b.batch * N;
    b.x_save += b.batch * N;
    b.out += b.batch * N;
    b.partial += grid * N;
  }
  return grad_h_tree(f->d_work, (float2 *)grad_H, N, l.sums, st, f->v.shape, LossSum{});
}

fft_status_t fft_filter_forward(fft_plan_t plan, const void *x, const void *H, void *y,
                                void *X_save, int conj_h, void *stream) {
  return filter_forward(plan, x, H, y, X_save, conj_h, true, stream);
}
fft_status_t fft_filter_forward_packed(fft_plan_t plan, const void *x, const void *H, void *y,
                                       void *X_packed, int conj_h, void *stream) {
  return filter_forward(plan, x, H, y, X_packed, conj_h, false, stream);
}
fft_status_t fft_filter_backward(fft_plan_t plan, const void *g_y, const void *H,
                                 const void *X_saved, void *grad_x, void *grad_H, void *stream) {
  return filter_backward(plan, g_y, H, X_saved, grad_x, grad_H, true, stream);
}
fft_status_t fft_filter_backward_packed(fft_plan_t plan, const void *g_y, const void *H,
                                        const void *X_packed, void *grad_x, void *grad_H,
                                        void *stream) {
  return filter_backward(plan, g_y, H, X_packed, grad_x, grad_H, false, stream);
}

fft_status_t fft_filter_step(fft_plan_t plan, const void *x, const void *H, const float *mask,
                             void *y, void *grad_x, void *grad_H, float *loss, void *stream) {
  fft_status_t s = filter_check(plan, x, H, grad_x);
  if (s != FFT_OK) return s;
  if (!mask || !grad_H || !loss) return FFT_ERR_INVALID_VALUE;
  if (((uintptr_t)mask | (uintptr_t)y | (uintptr_t)grad_H) & 15 || ((uintptr_t)loss & 3))
    return FFT_ERR_MISALIGNED;
  fft_plan_impl *pl = &plan->impl;
  FilterState *f = (FilterState *)pl->filter;
  cudaStream_t st = (cudaStream_t)stream;
  const int N = pl->N;
  if (pl->batch == 0) {
    if ((s = cuda_status(cudaMemsetAsync(grad_H, 0, sizeof(float2) * N, st))) != FFT_OK) return s;
    return cuda_status(cudaMemsetAsync(loss, 0, sizeof(float), st));
  }
  const int64_t bytes = (int64_t)sizeof(float2) * N * pl->batch;
  // Outputs: y and grad_x may each be x itself (a CTA reads its row before it
  // writes it) but overlap nothing else; the mask, H, grad_H and the loss
  // overlap no output.
  for (const void *o : {(const void *)y, (const void *)grad_x}) {
    if (!o) continue;
    if (o != x && overlap(o, bytes, x, bytes)) return FFT_ERR_INVALID_VALUE;
    if (overlap(o, bytes, mask, bytes / 2) || overlap(o, bytes, H, sizeof(float2) * N) ||
        overlap(o, bytes, grad_H, sizeof(float2) * N) || overlap(o, bytes, loss, sizeof(float)))
      return FFT_ERR_INVALID_VALUE;
  }
  if (y && overlap(y, bytes, grad_x, bytes)) return FFT_ERR_INVALID_VALUE;
  FilterStepArgs a{};
  a.x = (const float2 *)x;
  // grad_H may share memory with an input, which must stay until it is read
  const int64_t hb = (int64_t)sizeof(float2) * N;
  const bool own = overlap(grad_H, hb, H, hb) || overlap(grad_H, hb, x, bytes) ||
                   overlap(grad_H, hb, mask, bytes / 2);
  float2 *hp = own ? f->d_hp : (float2 *)grad_H;
  a.hp = hp;
  a.mask = mask;
  a.y = (float2 *)y;
  a.gx = (float2 *)grad_x;
  a.partial = f->d_work;
  a.loss_part = f->d_loss_part;
  a.tw = pl->d_tw;
  a.batch = pl->batch;
  a.inv_n = 1.0f / (float)N;
  const float2 *h = (const float2 *)H;
  int n = N;
  void *pack[] = {&h, &hp, &n, &f->v.shape};
  if ((s = cuda_status(launch_pdl((const void *)pack_h_kernel, dim3((N + 255) / 256), dim3(256), 0,
                                  st, pack))) != FFT_OK)
    return s;
  void *args[] = {&a};
  if ((s = cuda_status(launch_pdl(f->v.step.fn, dim3((unsigned)f->step_grid),
                                  dim3(f->v.threads), f->v.smem, st, args))) != FFT_OK)
    return s;
  return grad_h_tree(f->d_work, (float2 *)grad_H, N, f->step_grid, st, f->v.shape,
                     LossSum{f->d_loss_part, f->step_grid, loss});
}

}  // extern "C"
