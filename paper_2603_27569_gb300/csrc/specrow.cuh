// Row transforms for kernels that work on the spectrum inside the SM: the
// forward leaves the spectrum in the registers in an order of its own, the
// inverse starts from that order, and only the time-domain side is natural
// (thread lt of a row holds points lt + m T in register m, T = N / P).
//
// N = P T, T = RA RB.  Forward (decimation in frequency, Eq. 1 of the paper
// twice): with t = lt and k = k2 + P k1,
//   A[t][k2]  = W_N^{t k2} sum_m x[t + T m] W_P^{m k2}            (DFT_P)
//   X[k2 + P (k1a + RA k1b)] = sum_t A[t][k2] W_T^{t k1}, t = t0 + RB u:
//     sum_{t0} W_RB^{t0 k1b} W_T^{t0 k1a} sum_u A W_RA^{u k1a}    (DFT_RA, DFT_RB)
// The inverse runs the same steps backwards with conjugate roots.
//
// Why this order: after the first exchange (E1) every sub-row k2 belongs to
// one warp, so the second exchange (E2) and both exchanges of the inverse up
// to its last stay inside the warp's own rows of the buffer, and E1's
// time-domain side is written and read by the same thread.  A forward and
// inverse pair therefore needs two barriers of the row's threads (after E1's
// write, after the inverse's E1 write) and four exchanges, where two Stockham
// transforms that meet in natural order need five exchanges and ten barriers.
//
// Buffer: row k2 at k2 LDR; E1 keeps t at t, E2 keeps (t0, k1a) at t0 S + k1a.
// S = RA + 1 and LDR are odd-stepped so that every 8-byte access of a
// half-warp touches 16 distinct bank pairs.
//
// The twiddle rows sit in shared memory (TwRows of the schedule RB, RA, P,
// whose pass tables are exactly the two this transform needs): measured for
// one forward + inverse pair over 2^25 points, rows read through L1 / from
// shared memory: 16384 190 / 155, 8192 173 / 146, 4096 168 / 131, 1024
// 143 / 119 us (the streaming rows evict the tables: 13 % L1 hits).
//
// Packed order: register m of thread lt is entry ((m / 2) T + lt) 2 + (m & 1)
// of the row, so a saved spectrum moves in coalesced 16-byte accesses.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "stockham.cuh"

namespace fftgb {

// The packed order as plain numbers, for kernels that only move it.
struct SpecShape {
  int P, T, G, K, QB, RA, RB;  // P = 0: natural order
};
// Frequency held at entry pos of a packed row.
__host__ __device__ __forceinline__ int spec_freq(const SpecShape &s, int pos) {
  const int lt = (pos >> 1) % s.T, m = 2 * (pos / (2 * s.T)) + (pos & 1);
  const int e = (lt % s.G) * s.QB;
  return (lt / s.G) * s.K + e % s.K + s.P * (e / s.K) + m / s.RB + s.P * s.RA * (m % s.RB);
}

template <int N_, int P_, int RA_>
struct SpecRow {
  static constexpr int N = N_, P = P_, RA = RA_;
  static constexpr int T = N / P;    // threads per row, and length of a sub-row
  static constexpr int RB = T / RA;
  static constexpr int G = T < 32 ? T : 32;   // threads that share sub-rows
  static constexpr int K = G * P / T;         // sub-rows per group
  static constexpr int QA = P / RA, QB = P / RB;  // butterflies per thread
  static constexpr int S = RA + 1;
  static_assert(P * T == N && RA * RB == T && QA * RA == P && QB * RB == P, "sizes");
  static_assert(RB >= 16 && G % RB == 0 || RB == 32, "t0 does not depend on the butterfly");
  // smallest row pitch at which the E2 read (k2l fastest over the lanes) is
  // free of bank conflicts: QB LDR = 16 / (K / QB) modulo 16
  __host__ __device__ static constexpr int pitch() {
    int l = RA > 1 && RB * S > T ? RB * S : T;
    const int kk = K / QB > 16 ? 16 : K / QB;
    while ((QB * l) % 16 != (16 / kk) % 16) ++l;
    return l;
  }
  static constexpr int LDR = pitch();
  static constexpr int BUF = P * LDR;  // float2 per row
  // twiddle tables as a Stockham schedule RB, RA, P lays them out: pass 1 is
  // W_T^{t0 k1a}, the last pass W_N^{t k2}
  using Tables = std::conditional_t<(RA > 1), Sched<RB, RA, P>, Sched<RB, P>>;
  using Rows = TwRows<Tables, true>;
  static constexpr int TW = Rows::total();  // shared-memory entries
  static __host__ __device__ constexpr SpecShape shape() { return {P, T, G, K, QB, RA, RB}; }

  // The r - 1 twiddles of pass S at entry k, from the shared-memory rows.
  template <int S, int r, int p>
  static __device__ __forceinline__ void twiddles(float2 (&w)[r], const float2 *tw, int k) {
    const float2 *rows = tw + Rows::template offset<S>() + k;
#pragma unroll
    for (int j = 1; j < r; ++j)
      if (Rows::template loaded<r>(j)) w[j] = rows[Rows::template row<r>(j) * p];
    derive_from_pow2<r>(w);
  }

  // The row's threads meet: a warp, the whole CTA, or a named barrier.
  template <int TB>
  static __device__ __forceinline__ void row_sync(int b) {
    if constexpr (T <= 32) {
      __syncwarp();
    } else if constexpr (TB == 1) {
      __syncthreads();
    } else {
      asm volatile("bar.sync %0, %1;" ::"r"(b + 1), "n"(T) : "memory");
    }
  }

  // This thread's places in the buffer and in the spectrum.
  int lt, b;         // thread of the row, row of the CTA
  float2 *col;       // E1, time-domain side: column lt
  float2 *wa, *wb;   // the group's rows: DFT_RA side (t0), DFT_RB side (k2l, k1a)
  int t0;
  int k_base;        // frequency of spectrum register 0

  __device__ __forceinline__ SpecRow(float2 *buf, int lt_, int b_) : lt(lt_), b(b_) {
    const int gl = lt % G, wr = lt / G;
    col = buf + lt;
    t0 = gl % RB;
    wa = buf + (wr * K + gl / RB) * LDR + t0;
    const int e = gl * QB, k2l = e % K, k1a = e / K;
    wb = buf + (wr * K + k2l) * LDR + k1a;
    k_base = wr * K + k2l + P * k1a;
  }
  // Frequency of spectrum register m = q RB + k1b (q < QB): registers q = 0
  // and 1 hold adjacent frequencies.
  __device__ __forceinline__ int freq(int m) const {
    return k_base + m / RB + P * RA * (m % RB);
  }

  // offset of sub-row q of the DFT_RA side from wa
  static __device__ __forceinline__ constexpr int sub_a(int q) { return q * (G / RB) * LDR; }

  template <int TB>
  __device__ __forceinline__ void forward(float2 (&v)[P], const float2 *tw) const {
    Dft<P, -1>::run(v);
    {
      float2 w[P];
      twiddles<Tables::npass - 1, P, T>(w, tw, lt);
#pragma unroll
      for (int j = 1; j < P; ++j) v[j] = cmul(v[j], w[j]);
    }
#pragma unroll
    for (int j = 0; j < P; ++j) col[j * LDR] = v[j];
    row_sync<TB>(b);
    if constexpr (RA > 1) {
      float2 w[RA];
      twiddles<1, RA, RB>(w, tw, t0);
#pragma unroll
      for (int q = 0; q < QA; ++q)
#pragma unroll
        for (int u = 0; u < RA; ++u) v[q * RA + u] = wa[sub_a(q) + RB * u];
      __syncwarp();
#pragma unroll
      for (int q = 0; q < QA; ++q) {
        float2 d[RA];
#pragma unroll
        for (int u = 0; u < RA; ++u) d[u] = v[q * RA + u];
        Dft<RA, -1>::run(d);
#pragma unroll
        for (int j = 0; j < RA; ++j)
          wa[sub_a(q) + t0 * (S - 1) + j] = j ? cmul(d[j], w[j]) : d[j];
      }
      __syncwarp();
    }
#pragma unroll
    for (int q = 0; q < QB; ++q) {
      float2 d[RB];
#pragma unroll
      for (int i = 0; i < RB; ++i) d[i] = wb[q * LDR + (RA > 1 ? i * S : i)];
      Dft<RB, -1>::run(d);
#pragma unroll
      for (int i = 0; i < RB; ++i) v[q * RB + i] = d[i];
    }
  }

  template <int TB>
  __device__ __forceinline__ void inverse(float2 (&v)[P], const float2 *tw) const {
#pragma unroll
    for (int q = 0; q < QB; ++q) {
      float2 d[RB];
#pragma unroll
      for (int i = 0; i < RB; ++i) d[i] = v[q * RB + i];
      Dft<RB, +1>::run(d);
#pragma unroll
      for (int i = 0; i < RB; ++i) wb[q * LDR + (RA > 1 ? i * S : i)] = d[i];
    }
    if constexpr (RA > 1) {
      float2 w[RA];
      twiddles<1, RA, RB>(w, tw, t0);
      __syncwarp();
#pragma unroll
      for (int q = 0; q < QA; ++q) {
        float2 d[RA];
#pragma unroll
        for (int j = 0; j < RA; ++j) {
          d[j] = wa[sub_a(q) + t0 * (S - 1) + j];
          if (j) d[j] = cmulc(d[j], w[j]);
        }
        Dft<RA, +1>::run(d);
#pragma unroll
        for (int u = 0; u < RA; ++u) v[q * RA + u] = d[u];
      }
      __syncwarp();
#pragma unroll
      for (int q = 0; q < QA; ++q)
#pragma unroll
        for (int u = 0; u < RA; ++u) wa[sub_a(q) + RB * u] = v[q * RA + u];
    }
    row_sync<TB>(b);
    {
      float2 w[P];
      twiddles<Tables::npass - 1, P, T>(w, tw, lt);
#pragma unroll
      for (int j = 0; j < P; ++j) {
        v[j] = col[j * LDR];
        if (j) v[j] = cmulc(v[j], w[j]);
      }
    }
    Dft<P, +1>::run(v);
  }
};

}  // namespace fftgb
