// Column FFTs: batched length-L transforms down the columns of a row-major
// matrix, C adjacent columns per CTA.  This is the building block of the
// two-phase four-step path (paper Sec. IV-B, Eq. 3 and Sec. V-D):
//
//   N = N1 N2, input index n = n1 + N1 n2, output index k = k2 + N2 k1.
//   phase 1: for every n1, the N2-point FFT over n2 of x[n1 + N1 n2], times
//            the four-step twiddle W_N^{n1 k2}, stored as A[n1][k2];
//   phase 2: for every k2, the N1-point FFT over n1 of A[n1][k2], stored at
//            X[k2 + N2 k1].
//
// Both phases read C consecutive columns of every row, so each warp load
// covers whole row segments (128 bytes at C = 16; 32 bytes, one sector, at
// the narrowest C = 4).  In shared memory element (row, c) of the tile sits
// at row * C + c: with C = 16 a half-warp always touches 16 consecutive
// columns, so every exchange is free of bank conflicts without a swizzle.
// Phase 1 stores its result transposed (column-major).  From 256 points on
// the transpose is free: the last exchange is read with the threads dealt
// out the other way round (consecutive lanes take consecutive outputs of one
// column, from a padded tile), so the last pass leaves runs of T outputs per
// column in a warp and the store is coalesced.  (Measured over 2^25 points
// against one more trip through a padded tile, two barriers and 16 bytes of
// shared-memory traffic per point: row four-step 2^16 169 -> 158, 2^17 179 ->
// 167, 2^18 201 -> 183, 2^20 240 -> 221 us.)  Shorter phase 1s stage.
//
// Phase-1 twiddle W_N^{c k} for column c and output k: register m of thread
// lt holds k = lt + T m (T = L / P), so W_N^{c k} = W_N^{c lt} W_N^{c T m},
// the product of two exact table entries from grids laid out [c][lt] and
// [c][m]: a warp reads whole rows of the first and 16-byte pieces of one or
// two rows of the second instead of gathering one sector per element from a
// table of all N powers.  A staged phase 1, whose lanes hold consecutive
// columns, has them laid out [lt][c] and [m][c] (N = 4096 as 64 x 64: 159 us,
// with the other layout 193).
//
// Columns longer than one CTA holds (L = L1 L2 > 4096) run the same two
// phases down the column instead of along a row: input row n = n1 + L1 n2,
// output row k = k2 + L2 k1.  Phase 1 is an L2-point column FFT of each of the
// L1 sub-matrices n1 (rows n1, n1 + L1, ...), times W_L^{n1 k2}, the twiddle
// now indexed by the sub-matrix rather than the column (TWM == 2; a table
// laid out [n1][k2] of exact powers, one contiguous slice per CTA); phase 2
// is an L1-point column FFT of each of the L2 sub-matrices k2 of the phase-1
// result, stored to rows k2 + L2 k1.  A launch therefore covers nmat matrices
// of nsub sub-matrices each, sub-matrix j of matrix m starting at
// m * mat_stride + j * sub_stride.
#pragma once
#include "stockham.cuh"

namespace fftgb {

struct ColumnArgs {
  const float2 *in;
  float2 *out;
  const float2 *tw;      // per-pass tables of the length-L transform
  const float2 *tw_a;    // TWM 1: W_Ntot^{c lt} at c * T + lt (staged: lt * ncols + c);
                         // TWM 2: W_Ntot^{j k} at j * L + k for sub-matrix j; else null
  const float2 *tw_b;    // TWM 1: W_Ntot^{c T m} at c * P + m (staged: m * ncols + c)
  long long nmat;        // number of matrices times nsub
  long long in_mat_stride, out_mat_stride;  // elements between matrices
  long long in_sub_stride, out_sub_stride;  // elements between sub-matrices
  int nsub;              // sub-matrices per matrix (0 and 1: one)
  long long in_extent, out_extent;  // elements reachable from in / out (bounds-check build)
  int in_row_stride;     // elements between consecutive rows of the input
  int out_row_stride;    // elements between rows of a non-transposed output
  int ncols;             // columns per matrix (multiple of C)
  int ntot;              // L * ncols, the size of the four-step twiddle
  float scale;
};
struct ColumnLoopArgs : ColumnArgs {
  unsigned ntiles;  // tiles of the launch
};

// Row pitch of a tile that is read transposed, in its last exchange or staged:
// 16 consecutive lanes read outputs lt of one column at distinct bank pairs.
template <int C>
__host__ __device__ constexpr int transposed_pitch() {
  return C + 1;
}
// Does a phase 1 of L points read its last exchange transposed?  From 256
// points on, where a warp's runs are whole lines.  With the 64-byte runs of
// 128 points it gained 2 % at N = 8192..32768 but lost 5 % at 65536 (512 x
// 128: 174 / 183 us), and 17 % in the single-launch L2 form (167 / 195 us).
template <int L, int P, class SC>
__host__ __device__ constexpr bool merged_transpose() {
  return SC::npass > 1 && L / P >= 16;
}
// Padded tile: element (idx, c) at idx * LD + c.
template <int LD>
struct PaddedColumns {
  static constexpr int width = LD;
  int c;
  template <int p, int r>
  __device__ __forceinline__ int at(int idx) const { return idx * LD + c; }
};
// run_passes with the last exchange read by thread (lt2, c2) instead of (lt, c).
template <int L, int P, int D, class SC, int S, int LD>
__device__ __forceinline__ void run_passes_transposed(float2 (&a)[P], int lt, int c, int lt2,
                                                      int c2, float2 *buf,
                                                      const float2 *__restrict__ tw) {
  pass_compute<L, P, D, SC, S, 0>(a, lt, tw);
  if constexpr (S > 0) __syncthreads();  // every read of the buffer is done
  pass_write<L, P, SC, S>(a, lt, buf, PaddedColumns<LD>{c});
  __syncthreads();
  if constexpr (S + 2 == SC::npass) {
    pass_read<L, P, SC, S>(a, lt2, buf, PaddedColumns<LD>{c2});
    pass_compute<L, P, D, SC, S + 1, 0>(a, lt2, tw);
  } else {
    pass_read<L, P, SC, S>(a, lt, buf, PaddedColumns<LD>{c});
    run_passes_transposed<L, P, D, SC, S + 1, LD>(a, lt, c, lt2, c2, buf, tw);
  }
}
// Register m (output lt + T m of column col) times W_Ntot^{col (lt + T m)}.
template <int P, int T, int D>
__device__ __forceinline__ void phase1_twiddle(float2 (&a)[P], int lt, int col,
                                               const float2 *__restrict__ tw_a,
                                               const float2 *__restrict__ tw_b) {
  const float2 wa = __ldg(tw_a + (long long)col * T + lt);
  const float4 *wb = reinterpret_cast<const float4 *>(tw_b + (long long)col * P);
#pragma unroll
  for (int m = 0; m < P; m += 2) {
    const float4 w = __ldg(wb + m / 2);
    a[m] = cmul_dir<D>(a[m], cmul(wa, make_float2(w.x, w.y)));
    a[m + 1] = cmul_dir<D>(a[m + 1], cmul(wa, make_float2(w.z, w.w)));
  }
}

// The same where consecutive lanes hold consecutive columns (the staged
// transpose): grids laid out [lt][c] and [m][c].
template <int P, int D>
__device__ __forceinline__ void phase1_twiddle_staged(float2 (&a)[P], int lt, int col, int ncols,
                                                      const float2 *__restrict__ tw_a,
                                                      const float2 *__restrict__ tw_b) {
  const float2 wa = __ldg(tw_a + (long long)lt * ncols + col);
#pragma unroll
  for (int m = 0; m < P; ++m)
    a[m] = cmul_dir<D>(a[m], cmul(wa, __ldg(tw_b + (long long)m * ncols + col)));
}

// TWM: 0 no twiddle, 1 the row four-step's per-column twiddle (with a
// transposed store), 2 the per-sub-matrix twiddle of a long column.
template <int L, int P, int C, int D, class SC, int TWM, bool TRANSPOSED>
__global__ void __launch_bounds__(C *(L / P))
column_kernel(ColumnArgs args) {
  static_assert(SC::product() == L, "radix schedule must multiply to L");
  static_assert(P % SC::max_radix() == 0, "every radix must divide P");
  constexpr int T = L / P;
  constexpr int NT = C * T;
  extern __shared__ __align__(128) float2 smem[];
  // Programmatic dependent launch (see stockham_kernel): phase 2 may become
  // resident while phase 1 finishes, but reads nothing before it completed.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int c = threadIdx.x % C;
  const int lt = threadIdx.x / C;
  const int tiles_per_mat = args.ncols / C;
  const long long tile_mat = blockIdx.x / tiles_per_mat;
  const int c0 = (int)(blockIdx.x - tile_mat * tiles_per_mat) * C;
  long long mat = tile_mat, sub = 0;
  if (args.nsub > 1) {
    mat = tile_mat / args.nsub;
    sub = tile_mat - mat * args.nsub;
  }
  float2 a[P];
  {
    const long long base = mat * args.in_mat_stride + sub * args.in_sub_stride + c0 + c;
    const float2 *src = args.in + base;
#pragma unroll
    for (int m = 0; m < P; ++m) {
      const long long off = (long long)(lt + m * T) * args.in_row_stride;
      a[m] = FFTGB_OK(base + off, args.in_extent, kSiteColLoad) ? __ldg(src + off)
                                                               : make_float2(0.f, 0.f);
    }
  }
  if constexpr (TWM == 1 && TRANSPOSED && merged_transpose<L, P, SC>()) {
    const int lt2 = threadIdx.x % T, c2 = threadIdx.x / T;
    run_passes_transposed<L, P, D, SC, 0, transposed_pitch<C>()>(a, lt, c, lt2, c2, smem,
                                                                    args.tw);
    phase1_twiddle<P, T, D>(a, lt2, c0 + c2, args.tw_a, args.tw_b);
    const long long base = mat * args.out_mat_stride + (long long)(c0 + c2) * L + lt2;
    float2 *dst = args.out + base;
#pragma unroll
    for (int m = 0; m < P; ++m)  // final_index(lt2, m) = lt2 + T m
      if (FFTGB_OK(base + m * T, args.out_extent, kSiteColStore))
        dst[m * T] = cscale(a[m], args.scale);
    return;
  }
  run_passes<L, P, D, SC, 0>(a, lt, smem, args.tw, Interleaved<C>{c});
  // a[m] now holds output index final_index(lt, m) of column c0 + c.
  if constexpr (TWM == 1) {
    phase1_twiddle_staged<P, D>(a, lt, c0 + c, args.ncols, args.tw_a, args.tw_b);
  } else if constexpr (TWM == 2) {
    // W_L^{sub k}: the CTA reads one contiguous row of L entries, a warp at
    // most two adjacent entries per load (all C columns share k).
    const float2 *tw = args.tw_a + sub * L;
#pragma unroll
    for (int m = 0; m < P; ++m) {
      const int k = final_index<L, P, SC>(lt, m);
      if (FFTGB_OK(sub * L + k, (long long)(args.nsub > 1 ? args.nsub : 1) * L, kSiteColTwiddle))
        a[m] = cmul_dir<D>(a[m], __ldg(tw + k));
    }
  }
  if constexpr (TRANSPOSED) {
    // out[col * L + k]: stage through a padded tile.
    constexpr int LD = transposed_pitch<C>();
    __syncthreads();
#pragma unroll
    for (int m = 0; m < P; ++m) smem[final_index<L, P, SC>(lt, m) * LD + c] = a[m];
    __syncthreads();
    const long long base = mat * args.out_mat_stride + (long long)c0 * L;
    float2 *dst = args.out + base;
#pragma unroll
    for (int u = 0; u < P; ++u) {
      const int e = threadIdx.x + u * NT;  // e = col_local * L + k
      const int cl = e / L, k = e - cl * L;
      if (FFTGB_OK(base + e, args.out_extent, kSiteColStore))
        dst[e] = cscale(smem[k * LD + cl], args.scale);
    }
  } else {
    const long long base = mat * args.out_mat_stride + sub * args.out_sub_stride + c0 + c;
    float2 *dst = args.out + base;
#pragma unroll
    for (int m = 0; m < P; ++m) {
      const long long off = (long long)final_index<L, P, SC>(lt, m) * args.out_row_stride;
      if (FFTGB_OK(base + off, args.out_extent, kSiteColStore)) dst[off] = cscale(a[m], args.scale);
    }
  }
}

// Columns of 1024 to 4096 points, plain (no four-step twiddle, row-major
// store): the tile fills most of an SM, so one CTA per tile leaves the SM's
// loads, passes and stores one after the other.  Persistent instead: CTA c
// takes tiles c, c + G, ...; as it stores output register m it refills the
// register with the next tile's point m, and the tile's row segments were
// prefetched into L2 at the start of the tile before.  32 points per thread
// (128 registers: with 16 the loop's strided addresses spill).  Every twiddle
// row is read from a shared-memory copy made once per CTA.  Measured over
// 2^25 points, one CTA per tile with 16 points per thread / this: 1024
// 109 / 92 us with 16 columns, 99 with 8; 2048 137 / 122; 4096 (one launch)
// 188 / 164; as phase 2 of the row four-step 2^19 227 / 202, 2^20 257 / 242.
// Addresses are running pointers: per-point offsets from the strides measured
// 137 us at 2048.  What bounds it: one 16-warp CTA per SM, and at 2048 and 4096
// row segments of 64 and 32 bytes.
//
// First exchange (stride 1, radix r): thread lt writes rows lt r + j, so the
// 16 / C threads whose columns share a half-warp write rows r apart, the same
// banks.  Row x therefore sits at x ^ ((x / r) mod (16 / C)): the write's row
// becomes lt r + (j ^ (lt mod 16 / C)), and the read's lt + m T only depends
// on lt where T is a multiple of 16 r / C (checked), so both stay a per-thread
// base plus constants.
template <int L, int P, int C, int D, class SC, int S>
__device__ __forceinline__ void run_passes_shared(float2 (&a)[P], int lt, int c, float2 *buf,
                                                  const float2 *tw) {
  constexpr int r = SC::radix[S], p = SC::stride(S), T = L / P, Q = P / r;
  if constexpr (S > 0) {
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      const int k = (lt + q * T) & (p - 1);
      const bool ok = FFTGB_OK(k, p, kSiteTwiddle);
      const float2 *rows = tw + SC::tw_offset(S) + (ok ? k : 0);
#pragma unroll
      for (int j = 1; j < r; ++j) a[q + j * Q] = cmul_dir<D>(a[q + j * Q], rows[(j - 1) * p]);
    }
  }
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    float2 v[r];
#pragma unroll
    for (int j = 0; j < r; ++j) v[j] = a[q + j * Q];
    Dft<r, D>::run(v);
#pragma unroll
    for (int j = 0; j < r; ++j) a[q + j * Q] = v[j];
  }
  if constexpr (S + 1 < SC::npass) {
    if constexpr (S > 0) __syncthreads();  // every read of the buffer is done
    constexpr int share = 16 / C;  // rows of one half-warp
    if constexpr (S == 0 && share > 1) {
      static_assert(Q == 1 && r % share == 0, "one butterfly per thread, rows in groups");
      static_assert(T % r == 0, "(lt + m T) / r = lt / r + m T / r");
      const int x = lt & (share - 1);
#pragma unroll
      for (int j = 0; j < r; ++j) {
        const int row = lt * r + (j ^ x);
        if (FFTGB_OK(row, L, kSiteXchgWrite)) buf[row * C + c] = a[j];
      }
    } else {
      pass_write<L, P, SC, S>(a, lt, buf, Interleaved<C>{c});
    }
    __syncthreads();
    if constexpr (S == 0 && share > 1) {
#pragma unroll
      for (int m = 0; m < P; ++m) {
        // ((lt + m T) / r) mod share, m T / r known at compile time
        const int row = lt + m * T;
        const int at = row ^ ((lt / r + m * T / r) & (share - 1));
        a[m] = FFTGB_OK(at, L, kSiteXchgRead) ? buf[at * C + c] : make_float2(0.f, 0.f);
      }
    } else {
      pass_read<L, P, SC, S>(a, lt, buf, Interleaved<C>{c});
    }
    run_passes_shared<L, P, C, D, SC, S + 1>(a, lt, c, buf, tw);
  }
}

template <int L, int P, int C, int D, class SC>
__global__ void __launch_bounds__(C *(L / P), 65536 / (C * (L / P) * 128))
column_loop_kernel(ColumnLoopArgs args) {
  static_assert(SC::product() == L, "radix schedule must multiply to L");
  static_assert(P % SC::max_radix() == 0, "every radix must divide P");
  constexpr int T = L / P;
  constexpr int NT = C * T;
  extern __shared__ __align__(128) float2 smem[];
  float2 *tws = smem + L * C;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int c = threadIdx.x % C;
  const int lt = threadIdx.x / C;
  // element offset of tile t's first column, in the input or the output (the
  // launcher keeps tile numbers within 31 bits)
  const unsigned tiles_per_mat = args.ncols / C, nsub = args.nsub > 1 ? args.nsub : 1;
  auto base = [&](unsigned t, long long mat_stride, long long sub_stride) {
    const unsigned tm = t / tiles_per_mat, mat = tm / nsub;
    return mat * mat_stride + (tm - mat * nsub) * sub_stride + (t - tm * tiles_per_mat) * C;
  };
  const unsigned ntiles = args.ntiles;
  unsigned tile = blockIdx.x;
  float2 a[P];
  {
    const long long in = base(tile, args.in_mat_stride, args.in_sub_stride) + c;
#pragma unroll
    for (int m = 0; m < P; ++m) {
      const long long off = in + (long long)(lt + m * T) * args.in_row_stride;
      a[m] = FFTGB_OK(off, args.in_extent, kSiteColLoad) ? __ldg(args.in + off) : make_float2(0.f, 0.f);
    }
  }
  for (int i = threadIdx.x; i < SC::tw_total(); i += NT) tws[i] = __ldg(args.tw + i);
  // (published by the first exchange's barrier)
  for (; tile < ntiles; tile += gridDim.x) {
    const unsigned next = tile + gridDim.x;
    const bool load_next = next < ntiles;
    const long long in = load_next ? base(next, args.in_mat_stride, args.in_sub_stride) : 0;
    if (load_next) {
      for (int i = threadIdx.x; i < L; i += NT)
        if (FFTGB_OK(in + (long long)i * args.in_row_stride, args.in_extent, kSiteColLoad))
          asm volatile("prefetch.global.L2 [%0];" ::"l"(args.in + in +
                                                        (long long)i * args.in_row_stride));
    }
    // opaque per tile: nothing of the strides or the buffer is kept in
    // registers through the passes
    int zero = 0, ltp = lt, irs = args.in_row_stride, ors = args.out_row_stride;
    asm volatile("" : "+r"(zero), "+r"(ltp), "+r"(irs), "+r"(ors));
    run_passes_shared<L, P, C, D, SC, 0>(a, ltp, c, smem + zero, tws + zero);
    // register m is output row lt + m T (final_index) and input row lt + m T:
    // two running pointers
    const long long out = base(tile, args.out_mat_stride, args.out_sub_stride) + c;
    const float2 *src = args.in + (in + c + (long long)ltp * irs);
    float2 *dst = args.out + (out + (long long)ltp * ors);
    const long long istep = (long long)T * irs, ostep = (long long)T * ors;
#pragma unroll
    for (int m = 0; m < P; ++m) {
      static_assert(final_index<L, P, SC>(0, P - 1) == (P - 1) * T, "outputs are T rows apart");
      if (FFTGB_OK(dst - args.out, args.out_extent, kSiteColStore)) *dst = cscale(a[m], args.scale);
      dst += ostep;
      if (load_next) {
        a[m] = FFTGB_OK(src - args.in, args.in_extent, kSiteColLoad) ? __ldg(src)
                                                                     : make_float2(0.f, 0.f);
        src += istep;
      }
    }
    if (load_next) __syncthreads();  // the next tile rewrites the buffer
  }
}

}  // namespace fftgb
