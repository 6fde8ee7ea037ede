// Shared-memory FFT passes of the 2D transforms (fft.cuh holds the line transforms):
// the dense pass along x (rows), the dense pass along y (columns, in place) and the
// per-mode norms, with their tile shapes.  Included by the forward and the inverse
// translation units (fft_forward.cu, fft_inverse.cu).
#pragma once

#include <math.h>

#include <type_traits>

#include "fft.cuh"
#include "modes.cuh"
#include "pipeline.cuh"
#include "twofloat.cuh"

namespace fl {

namespace {

constexpr int THREADS = 256;  // of the single-pass (cluster) transforms

// ---- shapes of the dense passes --------------------------------------------------
// One butterfly of 16 (12) elements per thread in the first stage.  FP32 (bound by memory):
// tiles of up to 2048 elements in 128 threads, 16 loads in flight per thread and many CTAs
// per SM.  FP64 (bound by the FP64 pipe, which one warp per SM quarter fills): small tiles
// of 1-4 warps, so that the CTAs of a small problem spread over the SMs, and line counts
// that give every stage whole warps (a half-empty warp costs a whole one).
// T: fs_options.fft_tile (1: half the lines, radix cap 8)
constexpr int round32(int x) { return x <= 32 ? 32 : (x + 31) / 32 * 32; }
template <typename R, int N, int T> struct DensePass {
  static constexpr bool F32 = sizeof(R) == 4;
  static constexpr int MAXR = T == 0 ? 16 : 8;
  static constexpr int ROWS0 = F32 ? (N <= 16 ? 64 : N <= 32 ? 32 : N <= 128 ? 16 : 8)
                                   : (N == 8 ? 64 : N <= 16 ? 32 : N <= 32 ? 16 : N <= 192 ? 8 : 4);
  static constexpr int LINES = T == 0 ? ROWS0 : ROWS0 / 2;                            // rows per tile
  static constexpr int COLS = T == 0 ? (F32 || N <= 32 ? 16 : 8) : (F32 ? 8 : 4);     // columns per tile
  static constexpr int PT = T == 0 ? (N % 3 == 0 ? 12 : 16) : 8;                      // elements per thread
  static constexpr int threads(int lines) { return round32(lines * N / PT) < 256 ? round32(lines * N / PT) : 256; }
  static constexpr int RT = threads(LINES), CT = threads(COLS);
  static constexpr int SKEW = MAXR;
};

// CTAs per plane of the single-pass (cluster) transforms: the smallest power of two,
// at most 8 (the portable cluster size), that leaves each CTA at most 16 rows (24 for
// N = 192, 32 for N = 256)
template <int N, int MAXRB = 16> __host__ __device__ constexpr int plane_cluster() {
  int c = 1;
  while (c < 8 && N / c > MAXRB && N % (2 * c) == 0) c *= 2;
  return c;
}
// the one-pass forward transform's cluster: up to 32 rows per CTA (4 CTAs at N = 128;
// measured 2 us faster on the 128^2 step than 8 CTAs of 16 rows, and 16 CTAs of 8 rows
// slower still: fewer, larger tiles have less fixed cost)
template <int N> __host__ __device__ constexpr int fwd_cluster() { return plane_cluster<N, 32>(); }

template <typename R, int N>
__device__ __forceinline__ void load_twiddles(cx<R>* tw_s, const cx<R>* __restrict__ tw) {
  for (int j = threadIdx.x; j < N; j += THREADS) tw_s[j] = tw[j];
}

// Sum of |W|^2 over the n values of a block at src, from the NT threads' own sums q of squares, in
// two-float (the FP32 pipe): *out on thread 0.  Squares of values below 2^-63 leave the normal numbers of
// FP32, where those of W~, N to N^2 times larger, do not; a block whose threads' sums are all below
// 2^-64 reads its values again and takes them times SMALL_UNIT (its sum is below 2^-56 before, 2^112
// then).  Such a sum carries the minus sign, which squares have not; the classification joins the two
// kinds.  red: NT / 32 values.
template <int NT> __device__ __forceinline__ void block_sum_squares(float q, const float2* src, int n, ff* red,
                                                                    float2* out) {
  const bool unit = __syncthreads_or(!(q < 0x1p-64f)) != 0;  // (a NaN counts as one)
  if (!unit) {
    q = 0.f;
    for (int e = threadIdx.x; e < n; e += NT) {
      const float x = src[e].x * SMALL_UNIT, y = src[e].y * SMALL_UNIT;
      q += x * x + y * y;
    }
  }
  const ff s = ff_warp_sum(ff{q, 0.f});
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    ff t = red[0];
    for (int w = 1; w < NT / 32; ++w) t = ff_add(t, red[w]);
    *out = unit ? make_float2(t.hi, t.lo) : make_float2(-t.hi, -t.lo);
  }
}

// ---- dense pass along x (rows): forward, or inverse with 1/N^2 scaling --------
// grid (blocks, fields): field blockIdx.y has nrows rows.
// TI: element type of `in` (cx<R>, or float2 read into an FP64 transform); D32: FftPlan's
// factors in FP32 (IoPlan); WS (the data planes in FP32): also the block's sum of |in|^2 to wsum
// [field][block] (block_sum_squares).  clear (may be null): nclear words zeroed by block (0, 0), the counters of the
// classification that follows.
template <typename R, int N, bool INV, typename TI = cx<R>, int T = 0, bool D32 = false, bool WS = false>
__global__ void __launch_bounds__((DensePass<R, N, T>::RT))
k_fft_rows(const TI* __restrict__ in, cx<R>* out, long long nrows, const cx<R>* __restrict__ tw, R scale,
           unsigned* __restrict__ clear, int nclear, float2* __restrict__ wsum) {
  using DP = DensePass<R, N, T>;
  using PL = IoPlan<N, DP::MAXR, D32>;
  constexpr int LINES = DP::LINES;
  __shared__ cx<R> buf[PL::stages > 1 ? LayIdx<Lay::ROW, N, LINES, DP::SKEW>::ELEMS : 1];
  __shared__ cx<R> tws[PL::tw_elems];
  load_stage_twiddles<R, PL, N, DP::RT>(tws, tw);  // a constant table: read while the predecessor drains
  pdl_wait();
  pdl_trigger();
  if (clear && blockIdx.x == 0 && blockIdx.y == 0)
    for (int i = threadIdx.x; i < nclear; i += DP::RT) clear[i] = 0u;
  const long long row0 = (long long)blockIdx.x * LINES;
  const int rows = (int)(nrows - row0 < LINES ? nrows - row0 : LINES);
  const TI* src = in + (blockIdx.y * nrows + row0) * N;
  cx<R>* dst = out + (blockIdx.y * nrows + row0) * N;
  float ws = 0.f;
  fft_lines_io<R, PL, N, INV, LINES, DP::RT, Lay::ROW, DP::SKEW>(
      buf, tws,
      [&](int b, int i) {
        if (b >= rows) return czero<R>();
        if constexpr (WS) {
          const cx<R> v = src[b * N + i];
          ws += v.x * v.x + v.y * v.y;
          return v;
        } else if constexpr (std::is_same<TI, cx<R>>::value) {
          return src[b * N + i];
        } else {
          return from_d<R>(to_d(src[b * N + i]));
        }
      },
      [&](int b, int i, cx<R> v) {
        if (b < rows) dst[b * N + i] = INV ? scale * v : v;
      });
  if constexpr (WS) {
    __shared__ ff red[DP::RT / 32];
    block_sum_squares<DP::RT>(ws, src, rows * N, red, wsum + (long long)blockIdx.y * gridDim.x + blockIdx.x);
  }
}

// ---- dense pass along y (columns); grid (ceil(N/TC), planes); in == out is allowed ---
template <typename R, int N, bool INV, int T = 0, bool D32 = false>
__global__ void __launch_bounds__((DensePass<R, N, T>::CT))
k_fft_cols(const cx<R>* in, cx<R>* out, const cx<R>* __restrict__ tw) {
  using DP = DensePass<R, N, T>;
  using PL = IoPlan<N, DP::MAXR, D32>;
  constexpr int TC = DP::COLS;
  __shared__ cx<R> buf[PL::stages > 1 ? N * TC : 1];
  __shared__ cx<R> tws[PL::tw_elems];
  load_stage_twiddles<R, PL, N, DP::CT>(tws, tw);  // a constant table: read while the predecessor drains
  pdl_wait();
  pdl_trigger();
  const int c0 = blockIdx.x * TC;
  const long long o = (long long)blockIdx.y * N * N + c0;
  const cx<R>* src = in + o;
  cx<R>* dst = out + o;
  fft_lines_io<R, PL, N, INV, TC, DP::CT, Lay::COL, 0>(
      buf, tws, [&](int b, int i) { return N % TC == 0 || c0 + b < N ? src[i * N + b] : czero<R>(); },
      [&](int b, int i, cx<R> v) {
        if (N % TC == 0 || c0 + b < N) dst[i * N + b] = v;
      });
}

// ---- columns of the data planes and their norms in one pass ----------------------
// grid (ceil(N/TC), G, n_omega): block (tile, g, om) transforms its columns of the planes
// g ppg .. g ppg + ppg - 1 one after another and keeps sum |W~_k(nu)|^2 of its modes in
// registers (a thread's last-stage outputs are the same modes in every plane); gnorm [om][G][N^2]
// takes the sums, k_classify_early adds the groups.
// W~ is not written: it is needed only on the few columns that hold an active mode, and
// k_fft_cols_active transforms those again once they are known.  256 planes of 256^2 (FP32, bound
// by memory): columns 42 us + norms 32 us -> 30 us, and 14 us for the active columns.
// In FP64 the column pass is bound by the FP64 pipe and the norms run behind its tail: fused,
// with W~ written, 128^2 x 71 planes x 3 frequencies took 820 us for the whole call, 765 us with the
// two passes, so FP64 keeps those.
template <typename R, int N, int T>
__global__ void __launch_bounds__((DensePass<R, N, T>::CT))
k_fft_cols_norms(const cx<R>* __restrict__ wt, R* __restrict__ gnorm, int m1, int ppg, const cx<R>* __restrict__ tw) {
  using DP = DensePass<R, N, T>;
  using PL = IoPlan<N, DP::MAXR, false>;
  constexpr int TC = DP::COLS, CT = DP::CT, S = PL::stages - 1, RAD = PL::radix(S), NB = N / RAD;
  constexpr int PER = (TC * NB + CT - 1) / CT;
  __shared__ cx<R> buf[PL::stages > 1 ? N * TC : 1];
  __shared__ cx<R> tws[PL::tw_elems];
  load_stage_twiddles<R, PL, N, CT>(tws, tw);  // a constant table: read while the predecessor drains
  pdl_wait();
  pdl_trigger();
  const int c0 = blockIdx.x * TC, om = blockIdx.z;
  const int k0 = blockIdx.y * ppg, k1 = min(m1, k0 + ppg);
  R acc[PER][RAD];
#pragma unroll
  for (int p = 0; p < PER; ++p)
#pragma unroll
    for (int r = 0; r < RAD; ++r) acc[p][r] = R(0);
  for (int k = k0; k < k1; ++k) {
    const cx<R>* pl = wt + ((long long)om * m1 + k) * N * N + c0;
    auto ld = [&](int b, int i) { return N % TC == 0 || c0 + b < N ? pl[i * N + b] : czero<R>(); };
    if constexpr (S > 0) {
      if (k > k0) __syncthreads();  // the last plane's tile has been read
      io_first<R, PL, N, false, TC, CT, Lay::COL, 0>(buf, tws, ld);
    }
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      const int t = threadIdx.x + p * CT, b = t % TC, j = t / TC;  // as LayIdx<COL>::map
      if (TC * NB % CT == 0 || t < TC * NB) {
        cx<R> v[RAD];
        if constexpr (S > 0) {
          io_butterfly<R, PL, N, false, TC, Lay::COL, 0, S>(buf, tws, b, j, v);
        } else {
#pragma unroll
          for (int r = 0; r < RAD; ++r) v[r] = ld(b, r);
          Dft<R, false>::template run<RAD>(v);
        }
#pragma unroll
        for (int r = 0; r < RAD; ++r) acc[p][r] += v[r].x * v[r].x + v[r].y * v[r].y;
      }
    }
  }
  R* g = gnorm + ((long long)om * gridDim.y + blockIdx.y) * N * N + c0;
#pragma unroll
  for (int p = 0; p < PER; ++p) {
    const int t = threadIdx.x + p * CT, b = t % TC, j = t / TC;
    if ((TC * NB % CT == 0 || t < TC * NB) && (N % TC == 0 || c0 + b < N))
#pragma unroll
      for (int r = 0; r < RAD; ++r) g[(j + r * NB) * N + b] = acc[p][r];
  }
}

// the columns of the compact list of frequency om (those that hold an active mode), in place on
// the row-transformed planes: 4 columns by 4 planes per tile, as k_ifft_cols_gather
template <typename R, int N> struct ActivePass {
  static constexpr int GC = 4, GL = 4, LINES = GC * GL;
  using PL = IoPlan<N, 16, false>;
  static constexpr int NT = round32(LINES * N / (N % 3 == 0 ? 12 : 16)) < 256 ? round32(LINES * N / (N % 3 == 0 ? 12 : 16)) : 256;
};
template <typename R, int N>
__global__ void __launch_bounds__((ActivePass<R, N>::NT))
k_fft_cols_active(cx<R>* wt, int m1, const unsigned* __restrict__ colmask, const cx<R>* __restrict__ tw) {
  using AP = ActivePass<R, N>;
  using PL = typename AP::PL;
  constexpr int GC = AP::GC, GL = AP::GL;
  __shared__ cx<R> buf[PL::stages > 1 ? N * AP::LINES : 1];
  __shared__ cx<R> tws[PL::tw_elems];
  __shared__ short cols[N];
  load_stage_twiddles<R, PL, N, AP::NT>(tws, tw);
  pdl_wait();
  pdl_trigger();
  // the list of the columns, from their mask
  int nc = 0;
  {
    const unsigned* cm = colmask + 8 * blockIdx.y;
    for (int i = threadIdx.x; i < N; i += AP::NT) {
      int at = 0;
      for (int w = 0; w < i / 32; ++w) at += __popc(cm[w]);
      const unsigned m = cm[i / 32];
      if (m >> (i & 31) & 1u) cols[at + __popc(m & ((1u << (i & 31)) - 1u))] = (short)i;
    }
    for (int w = 0; w < (N + 31) / 32; ++w) nc += __popc(cm[w]);
    __syncthreads();
  }
  const int om = blockIdx.y, k0 = blockIdx.x * GL;
  const int nk = min(GL, m1 - k0);
  cx<R>* pl = wt + ((long long)om * m1 + k0) * N * N;
  for (int cb = blockIdx.z * GC; cb < nc; cb += gridDim.z * GC) {
    if (cb != (int)blockIdx.z * GC) __syncthreads();  // the previous tile has been read
    const int ncb = min(GC, nc - cb);
    const short* cl = cols + cb;
    // line b: column b % GC, plane b / GC (neighbouring columns are mostly neighbours in a row)
    fft_lines_io<R, PL, N, false, AP::LINES, AP::NT, Lay::COL, 0>(
        buf, tws,
        [&](int b, int i) {
          return b % GC < ncb && b / GC < nk ? pl[((long long)(b / GC) * N + i) * N + cl[b % GC]] : czero<R>();
        },
        [&](int b, int i, cx<R> v) {
          if (b % GC < ncb && b / GC < nk) pl[((long long)(b / GC) * N + i) * N + cl[b % GC]] = v;
        });
  }
}

// ---- per-mode norms ||W~_nu||^2 = sum_k |W~_k(nu)|^2 ----------------------------
// grid (n_partial, n_omega), NORM_MB modes per block and NORM_Q threads per mode: warp
// w sums the planes of quarter q = w / 2 (a contiguous quarter of the planes, its loads
// in flight together) for 32 consecutive modes, and the quarters are added in a fixed
// order; each block also writes the sum of its modes' norms (fixed-order tree) for ||W||.
constexpr int NORM_T = 256, NORM_Q = 4, NORM_MB = NORM_T / NORM_Q;

template <typename R>
__global__ void __launch_bounds__(NORM_T)
k_mode_norms(const cx<R>* __restrict__ wt, double* __restrict__ norms, double* __restrict__ partial, int m1,
             int N2, unsigned long long* __restrict__ ctr) {
  pdl_wait();
  pdl_trigger();
  __shared__ R part[NORM_Q][NORM_MB];
  __shared__ double red[NORM_MB];
  const int om = blockIdx.y;
  const int q = threadIdx.x / NORM_MB, j = threadIdx.x % NORM_MB;
  const int nu = blockIdx.x * NORM_MB + j;
  // summed in the working precision R (FP32 in the mixed path: FP64 arithmetic
  // here would run on the slow FP64 pipe for every mode)
  R acc = R(0);
  const int k0 = q * m1 / NORM_Q, k1 = (q + 1) * m1 / NORM_Q;
  if (nu < N2) {
    const cx<R>* p = wt + (long long)om * m1 * N2 + nu;
    int k = k0;
    for (; k + 8 <= k1; k += 8) {  // eight independent loads in flight, summed in plane order
      cx<R> v[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) v[t] = p[(long long)(k + t) * N2];
#pragma unroll
      for (int t = 0; t < 8; ++t) acc += v[t].x * v[t].x + v[t].y * v[t].y;
    }
    for (; k < k1; ++k) {
      const cx<R> v = p[(long long)k * N2];
      acc += v.x * v.x + v.y * v.y;
    }
  }
  part[q][j] = acc;
  __syncthreads();
  R nrm = R(0);
  if (q == 0) {
    nrm = (part[0][j] + part[1][j]) + (part[2][j] + part[3][j]);
    if (nu < N2) norms[(long long)om * N2 + nu] = (double)nrm;
    red[j] = (double)nrm;
  }
  // modes whose norm is not finite (a NaN or Inf in W), counted at the barrier
  // the reduction needs anyway
  const int n_bad = __syncthreads_count(q == 0 && nu < N2 && !isfinite(nrm));
  if (n_bad && threadIdx.x == 0) atomicAdd(ctr + C_NONFINITE, (unsigned long long)n_bad);
  for (int h = NORM_MB / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[(long long)om * gridDim.x + blockIdx.x] = red[0];
}

}  // namespace

#define FL_SIZES(X) X(8) X(12) X(16) X(24) X(32) X(48) X(64) X(96) X(128) X(192) X(256)

}  // namespace fl
