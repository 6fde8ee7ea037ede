// Forward 2D FFT passes of Algorithm 2 (step 1) and the dense 2D transforms of the
// forward solvers and derivatives, for N = 2^a 3^b <= 256, in FP64 (double2) or FP32
// (float2).
//
//   fft2_forward  : W -> W~ on every data plane (Sec. 4, Algorithm 2 step 1 needs
//                   W~ = F_r[W]), then ||W~_nu||^2 summed over the planes of a
//                   frequency, which the discrepancy test needs (FP32: in the
//                   classification, from ||W||^2 summed here over W itself).
//   real planes   : F_r[xi] of the plane-wave generator; rows around the product
//                   with xi of Algorithm 1's iteration; the inverse rows of the
//                   derivatives' directions joined with step 3.
// The inverse passes of a reconstruction are in fft_inverse.cu.
#include "diff.cuh"
#include "fft_pass.cuh"

namespace fl {

namespace {

template <typename R>
__global__ void k_twiddles(cx<R>* tw, int n) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n) {
    double s, c;
    sincospi(-2.0 * (double)j / (double)n, &s, &c);
    tw[j] = from_d<R>(make_double2(c, s));
  }
}

// ---- single-pass forward 2D transform: one data plane per cluster ------------------
// grid (C, planes), clusters of C = fwd_cluster<N>() CTAs along x.  CTA r of the
// cluster of plane p loads rows r RB .. r RB + RB - 1 (RB = N / C) of the plane into
// its shared memory and transforms them along x; after a cluster barrier it reads
// columns r RB .. r RB + RB - 1 of all N rows from the CTAs that hold them
// (distributed shared memory), transforms them along y and writes them to W~.  The
// plane crosses global memory once each way, in one launch.
// clear (may be null): nclear words zeroed by CTA (0, 0), as in k_fft_rows.
template <typename R, int N> __host__ __device__ constexpr size_t plane_fwd_smem() {
  constexpr int RB = N / fwd_cluster<N>();
  return sizeof(cx<R>) * ((size_t)LayIdx<Lay::ROW, N, RB, 16>::ELEMS + (size_t)RB * N + N);
}

// wsum (may be null): the CTA's sum of |in|^2, [plane][C] (block_sum_squares).
template <typename R, int N>
__global__ void __launch_bounds__(THREADS)
k_fft2_plane(const cx<R>* __restrict__ in, cx<R>* __restrict__ out, const cx<R>* __restrict__ tw,
             unsigned* __restrict__ clear, int nclear, float2* __restrict__ wsum) {
  constexpr int C = fwd_cluster<N>(), RB = N / C;
  using IA = LayIdx<Lay::ROW, N, RB, 16>;  // this CTA's rows
  constexpr int E = RB * N;                // elements of the row tile and of the column tile
  constexpr int PER = (E + THREADS - 1) / THREADS;
  extern __shared__ __align__(16) unsigned char plane_smem[];
  cx<R>* rows = reinterpret_cast<cx<R>*>(plane_smem);
  cx<R>* colt = rows + IA::ELEMS;  // column tile: element i of column b at i RB + b
  cx<R>* tw_s = colt + E;
  const unsigned r = cluster_rank();
  load_twiddles<R, N>(tw_s, tw);  // a constant table: read while the predecessor drains
  pdl_wait();
  pdl_trigger();
  if (clear && blockIdx.x == 0 && blockIdx.y == 0)
    for (int i = threadIdx.x; i < nclear; i += THREADS) clear[i] = 0u;
  const long long pb = (long long)blockIdx.y * N * N;
  const cx<R>* src = in + pb + (long long)r * E;
  cx<R> v[PER];
#pragma unroll
  for (int p = 0; p < PER; ++p) {
    const int e = threadIdx.x + p * THREADS;
    if (E % THREADS == 0 || e < E) v[p] = src[e];
  }
  float ws = 0.f;
#pragma unroll
  for (int p = 0; p < PER; ++p)
    if (E % THREADS == 0 || threadIdx.x + p * THREADS < E) ws += v[p].x * v[p].x + v[p].y * v[p].y;
#pragma unroll
  for (int p = 0; p < PER; ++p) {
    const int e = threadIdx.x + p * THREADS;
    if (E % THREADS == 0 || e < E) rows[IA::at(e / N, e % N)] = v[p];
  }
  __syncthreads();
  fft_lines<R, N, false, RB, THREADS, Lay::ROW, 16, 16>(rows, tw_s);
  cluster_sync();  // every CTA's rows are transformed
  // row i of column r RB + b sits in row i % RB of CTA i / RB: all loads first, then
  // the stores, so that the remote loads overlap
#pragma unroll
  for (int p = 0; p < PER; ++p) {
    const int e = threadIdx.x + p * THREADS;
    if (E % THREADS == 0 || e < E) {
      const int i = e / RB, b = e - (e / RB) * RB;
      v[p] = dsmem_ld(dsmem_addr(rows + IA::at(i % RB, (int)r * RB + b), (unsigned)(i / RB)), v[p]);
    }
  }
#pragma unroll
  for (int p = 0; p < PER; ++p) {
    const int e = threadIdx.x + p * THREADS;
    if (E % THREADS == 0 || e < E) colt[e] = v[p];
  }
  cluster_arrive();  // this CTA has read the others' rows
  __syncthreads();
  fft_lines<R, N, false, RB, THREADS, Lay::COL, 16>(colt, tw_s);
  cx<R>* dst = out + pb + (long long)r * RB;
#pragma unroll
  for (int p = 0; p < PER; ++p) {
    const int e = threadIdx.x + p * THREADS;
    if (E % THREADS == 0 || e < E) dst[(long long)(e / RB) * N + e % RB] = colt[e];
  }
  if (wsum) {
    __shared__ ff red[THREADS / 32];
    block_sum_squares<THREADS>(ws, src, E, red, wsum + (long long)blockIdx.y * C + r);
  }
  cluster_wait();  // no CTA leaves while another may still read its rows
}

template <typename R, int N>
cudaError_t fwd_plane(const cx<R>* W, const Problem& P, const Work<R>& w, cudaStream_t s, cudaEvent_t mid,
                      bool norms, int* n_wsum) {
  constexpr size_t smem = plane_fwd_smem<R, N>();
  static SmemOptIn attr;
  cudaError_t e = opt_in_smem(attr, (const void*)k_fft2_plane<R, N>, smem, true);
  if (e != cudaSuccess) return e;
  constexpr int C = fwd_cluster<N>();
  const bool early = norms && classify_early(P, sizeof(R) == 8);
  if (early) *n_wsum = C * P.m1;
  e = launch_pdl_cluster(k_fft2_plane<R, N>, dim3(C, (unsigned)(P.n_omega * P.m1)), dim3(THREADS), C, smem, s, W,
                         w.wt, (const cx<R>*)w.tw, w.bar, clear_words(P), early ? w.wsum : (float2*)nullptr);
  if (e != cudaSuccess) return e;
  if (mid) cudaEventRecord(mid, s);
  if (early || !norms) return cudaGetLastError();
  return launch_mode_norms<R>(P, w, s);
}

// ---- real planes -------------------------------------------------------------------
// Rows: the forward transform along x of real rows, two neighbours (2y, 2y + 1) of one plane to a
// complex line: with Z their joint transform, twice the two are Z_k + conj(Z_{N-k}) and
// -i (Z_k - conj(Z_{N-k})), taken apart behind the last stage.  Two PLANES to a line would cost the
// same, but then the weaker plane's transform carries the stronger one's rounding.  out [plane][N][N/2 + 2]
// holds the columns k <= N/2 (the rest are their mirror images) and one more, for whole 32-byte
// sectors.
template <typename R, int N>
__global__ void __launch_bounds__((DensePass<R, N, 0>::RT))
k_fft_rows_real(const R* __restrict__ xi, cx<R>* __restrict__ out, long long npairs, const cx<R>* __restrict__ tw) {
  using DP = DensePass<R, N, 0>;
  using PL = IoPlan<N, DP::MAXR, false>;
  constexpr int LINES = DP::LINES, HS = real_stride(N);
  using IX = LayIdx<Lay::ROW, N, LINES, DP::SKEW>;
  static_assert(N % 2 == 0, "a pair of rows lies in one plane");
  __shared__ cx<R> buf[IX::ELEMS];
  __shared__ cx<R> tws[PL::tw_elems];
  load_stage_twiddles<R, PL, N, DP::RT>(tws, tw);
  pdl_wait();
  pdl_trigger();
  const long long p0 = (long long)blockIdx.x * LINES;
  const int np = (int)(npairs - p0 < LINES ? npairs - p0 : LINES);
  const R* src = xi + 2 * p0 * N;
  cx<R>* dst = out + 2 * p0 * HS;
  fft_lines_io<R, PL, N, false, LINES, DP::RT, Lay::ROW, DP::SKEW>(
      buf, tws,
      [&](int b, int i) { return b < np ? mk<R>(src[2 * b * N + i], src[(2 * b + 1) * N + i]) : czero<R>(); },
      [&](int b, int i, cx<R> v) { buf[IX::at(b, i)] = v; });
  __syncthreads();
  for (int e = threadIdx.x; e < np * HS; e += DP::RT) {
    const int b = e / HS, k = e % HS;
    const cx<R> z = buf[IX::at(b, k)], c = buf[IX::at(b, k == 0 ? 0 : N - k)];
    dst[2 * b * HS + k] = mk<R>(z.x + c.x, z.y - c.y);
    dst[(2 * b + 1) * HS + k] = mk<R>(z.y + c.y, c.x - z.x);
  }
}

// Columns: the columns k <= N/2 of every plane in place, a tile any COLS consecutive ones of the
// M (N/2 + 1), so that the odd one of a plane fills no tile of its own (FP64, 37 planes of 192^2: 481
// tiles plane by plane, a fourth one on some of the SMs, and 449 these)
template <typename R, int N>
__global__ void __launch_bounds__((DensePass<R, N, 0>::CT))
k_fft_cols_real(cx<R>* data, int ncols, const cx<R>* __restrict__ tw) {
  using DP = DensePass<R, N, 0>;
  using PL = IoPlan<N, DP::MAXR, false>;
  constexpr int TC = DP::COLS, H = N / 2 + 1, HS = real_stride(N);
  static_assert(DP::CT % TC == 0, "a thread stays in its column");
  __shared__ cx<R> buf[PL::stages > 1 ? N * TC : 1];
  __shared__ cx<R> tws[PL::tw_elems];
  load_stage_twiddles<R, PL, N, DP::CT>(tws, tw);
  pdl_wait();
  pdl_trigger();
  const int q = blockIdx.x * TC + threadIdx.x % TC;
  const bool on = q < ncols;
  cx<R>* col = data + (on ? (long long)(q / H) * N * HS + q % H : 0);
  fft_lines_io<R, PL, N, false, TC, DP::CT, Lay::COL, 0>(
      buf, tws, [&](int, int i) { return on ? col[i * HS] : czero<R>(); },
      [&](int, int i, cx<R> v) {
        if (on) col[i * HS] = v;
      });
}

// ---- rows: inverse along x, times xi, forward along x --------------------------------
// The middle of F[xi F^-1 U~]: between the two column passes everything happens within a
// row, so one kernel reads and writes the planes once.  The product happens between the two
// transforms' registers: outputs j + r N/R1 of the last inverse stage (radix R1) for j = k, k + N/R0, ..
// are the inputs k + r N/R0 of butterfly k of the first forward stage (radix R0) when R1 divides R0, and
// a thread that runs those R0/R1 inverse butterflies goes on with the forward one.  Other plans write
// the product to the tile in place, from registers.  Either way the kernel needs one tile: a second
// one for the product left five 64-thread blocks per SM at N = 128 in FP64 (86 registers), and one more
// crossing.  Bound by the FP64 pipe: 128^2 x 64 FP64 110 us -> 96 us (85% of that pipe's rate).
template <typename R, int N> struct RowsXi {
  using DP = DensePass<R, N, 0>;
  using PL = IoPlan<N, DP::MAXR, sizeof(R) == 4>;
  using IX = LayIdx<Lay::ROW, N, DP::LINES, DP::SKEW>;
  static constexpr int S = PL::stages - 1, R0 = PL::radix(0), R1 = PL::radix(S);
  static constexpr bool REG = S == 1 && R0 % R1 == 0;
};
template <typename R, int N>
__global__ void __launch_bounds__((DensePass<R, N, 0>::RT))
k_rows_xi(cx<R>* __restrict__ data, const R* __restrict__ xi, long long nrows, const cx<R>* __restrict__ tw,
          R scale) {
  using RX = RowsXi<R, N>;
  using DP = typename RX::DP;
  using PL = typename RX::PL;
  using IX = typename RX::IX;
  constexpr int LINES = DP::LINES, NT = DP::RT, SK = DP::SKEW, S = RX::S, R0 = RX::R0, R1 = RX::R1;
  extern __shared__ __align__(16) unsigned char rows_xi_smem[];  // IX::ELEMS elements
  cx<R>* buf = reinterpret_cast<cx<R>*>(rows_xi_smem);
  __shared__ cx<R> tws[PL::tw_elems];
  load_stage_twiddles<R, PL, N, NT>(tws, tw);
  pdl_wait();
  pdl_trigger();
  const long long row0 = (long long)blockIdx.x * LINES;
  const int rows = (int)(nrows - row0 < LINES ? nrows - row0 : LINES);
  cx<R>* d = data + row0 * N;
  const R* x = xi + row0 * N;
  auto ld = [&](int b, int i) { return b < rows ? d[b * N + i] : czero<R>(); };
  auto st = [&](int b, int i, cx<R> v) {
    if (b < rows) d[b * N + i] = v;
  };
  auto ldx = [&](int b, int i) { return b < rows ? scale * x[b * N + i] : R(0); };
  if constexpr (S == 0) {  // a thread owns whole lines
    for (int b = threadIdx.x; b < rows; b += NT) {
      cx<R> v[R0];
#pragma unroll
      for (int r = 0; r < R0; ++r) v[r] = ld(b, r);
      Dft<R, true>::template run<R0>(v);
#pragma unroll
      for (int r = 0; r < R0; ++r) v[r] = ldx(b, r) * v[r];
      Dft<R, false>::template run<R0>(v);
#pragma unroll
      for (int r = 0; r < R0; ++r) st(b, r, v[r]);
    }
  } else {
    io_first<R, PL, N, true, LINES, NT, Lay::ROW, SK>(buf, tws, ld);
    // the last inverse stage and the product; in place once every thread has read its inputs
    constexpr int RAD = RX::REG ? R0 : R1, NB = N / RAD, TOTAL = LINES * NB, PER = (TOTAL + NT - 1) / NT;
    cx<R> v[PER][RAD];
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      const int t = threadIdx.x + p * NT;
      if (TOTAL % NT == 0 || t < TOTAL) {
        int b, k;
        IX::map(t, NB, b, k);
        R f[RAD];
#pragma unroll
        for (int r = 0; r < RAD; ++r) f[r] = ldx(b, k + r * NB);
        constexpr int Q = RAD / R1;  // inverse butterflies k, k + NB, ..
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          cx<R> y[R1];
          io_butterfly<R, PL, N, true, LINES, Lay::ROW, SK, S>(buf, tws, b, k + q * NB, y);
#pragma unroll
          for (int r = 0; r < R1; ++r) v[p][q + r * Q] = f[q + r * Q] * y[r];
        }
        if constexpr (RX::REG) Dft<R, false>::template run<R0>(v[p]);
      }
    }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      const int t = threadIdx.x + p * NT;
      if (TOTAL % NT == 0 || t < TOTAL) {
        int b, k;
        IX::map(t, NB, b, k);
#pragma unroll
        for (int r = 0; r < RAD; ++r) buf[IX::at(b, RX::REG ? k * R0 + r : k + r * NB)] = v[p][r];
      }
    }
    __syncthreads();
    if constexpr (!RX::REG)
      io_first<R, PL, N, false, LINES, NT, Lay::ROW, SK, false, true>(
          buf, tws, [&](int b, int i) { return buf[IX::at(b, i)]; });
    io_last<R, PL, N, false, LINES, NT, Lay::ROW, SK>(buf, tws, st);
  }
}

// ---- inverse rows of a direction's fields with the derivative of step 3 ----------
// Block (d, b): LINES rows of X of direction d; for every frequency the rows of dV~ and dU~ are
// transformed along x in the tile and each thread adds its voxels' terms
//   num = Re(conj(du) V + conj(u) dV),  dD = 2 Re(conj(u) du),  D = |u|^2
// with V and u of the tape (the directions of a row block run side by side and share them in
// L2): dxi = (num - xi dD) / D.  Writing dV and du and reading them back for a pointwise kernel took
// 2.1 of 6.5 GB of a 16-direction call at 128^2 x 64, 4 frequencies (FP32): rows 307 us + point
// 212 us before, 417 us now.  In FP32 V and u are loaded before the rows are transformed, and
// 256 threads share a tile from N = 96 on, so that more loads are in flight (420 us without the
// first at 128 threads, 436 us with it).  16 directions, 32 planes, 2 frequencies, with 128 threads beside:
// N = 128 133 us (147), but 96 120 (111) and 192 640 (510), whose 12-point last stage leaves 256 threads
// idle in part; below, 128 against 256: 32 12.0 (14.2), 48 19.6 (23.2), 64 32.9 (33.2).
template <typename R, int N> struct JvpPass {
  static constexpr bool F32 = sizeof(R) == 4;
  using PL = IoPlan<N, F32 || N != 256 ? 16 : 8, F32>;
  static constexpr int NT = F32 ? (N >= 96 ? 256 : 128) : (N >= 192 ? 128 : 64);
  static constexpr int LINES = F32 ? (N <= 16 ? 16 : 8) : (N <= 16 ? 8 : 4);
  static constexpr int E = LINES * N, PER = (E + NT - 1) / NT;
  using IX = LayIdx<Lay::ROW, N, 2 * LINES, 16>;
};
template <typename R, int N>
__global__ void __launch_bounds__((JvpPass<R, N>::NT))
k_jvp_rows(Problem P, const cx<R>* __restrict__ dv, const cx<R>* __restrict__ du, const cx<R>* __restrict__ Vx,
           const cx<R>* __restrict__ ux, const R* __restrict__ xis, R* __restrict__ dxi, const cx<R>* __restrict__ tw) {
  using JP = JvpPass<R, N>;
  using PL = typename JP::PL;
  using IX = typename JP::IX;
  constexpr int LINES = JP::LINES, NT = JP::NT, E = JP::E, PER = JP::PER;
  constexpr int PRE = JP::F32 ? PER : 0;  // FP64: no registers to spare
  __shared__ cx<R> buf[IX::ELEMS];
  __shared__ cx<R> tws[PL::tw_elems];
  load_stage_twiddles<R, PL, N, NT>(tws, tw);
  pdl_wait();
  pdl_trigger();
  const long long nrows = (long long)P.m * N, MN2 = nrows * N;
  const long long row0 = (long long)blockIdx.y * LINES;
  const int rows = (int)(nrows - row0 < LINES ? nrows - row0 : LINES);
  const R scale = R(P.inv_n2), guard2 = R(P.u_guard);
  R num[PER], dD[PER], D[PER];
#pragma unroll
  for (int p = 0; p < PER; ++p) num[p] = dD[p] = D[p] = R(0);
  for (int om = 0; om < P.n_omega; ++om) {
    const long long at = ((long long)blockIdx.x * P.n_omega + om) * MN2 + row0 * N;
    const cx<R>*a = dv + at, *b = du + at;
    const cx<R>*V = Vx + om * MN2 + row0 * N, *u = ux + om * MN2 + row0 * N;
    cx<R> pv[PRE + 1], pu[PRE + 1];  // on their way while the rows are transformed
#pragma unroll
    for (int p = 0; p < PRE; ++p) {
      const int e = threadIdx.x + p * NT;
      pv[p] = e < rows * N ? V[e] : czero<R>();
      pu[p] = e < rows * N ? u[e] : czero<R>();
    }
    if (om > 0) __syncthreads();  // the tile has been read
    fft_lines_io<R, PL, N, true, 2 * LINES, NT, Lay::ROW, 16>(
        buf, tws,
        [&](int line, int i) {
          const int bl = line >= LINES ? line - LINES : line;
          return bl < rows ? (line >= LINES ? b : a)[bl * N + i] : czero<R>();
        },
        [&](int line, int i, cx<R> v) { buf[IX::at(line, i)] = v; });
    __syncthreads();
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      const int e = threadIdx.x + p * NT;
      if (e < rows * N) {
        const cx<R> x = scale * buf[IX::at(e / N, e % N)], y = scale * buf[IX::at(LINES + e / N, e % N)];
        const cx<R> v = p < PRE ? pv[p] : V[e], w = p < PRE ? pu[p] : u[e];
        num[p] += y.x * v.x + y.y * v.y + w.x * x.x + w.y * x.y;
        dD[p] += R(2) * (w.x * y.x + w.y * y.y);
        D[p] += abs2(w);
      }
    }
  }
#pragma unroll
  for (int p = 0; p < PER; ++p) {
    const int e = threadIdx.x + p * NT;
    if (e < rows * N) {
      const long long o = row0 * N + e;
      dxi[blockIdx.x * MN2 + o] = D[p] < guard2 ? R(0) : (num[p] - xis[o] * dD[p]) / D[p];
    }
  }
}

template <typename R, int N, bool INV, typename TI, int T, bool D32>
cudaError_t rows_launch(const TI* in, cx<R>* out, long long nrows, const cx<R>* tw, R scale, cudaStream_t s) {
  using DP = DensePass<R, N, T>;
  return launch_pdl(k_fft_rows<R, N, INV, TI, T, D32>, dim3((unsigned)((nrows + DP::LINES - 1) / DP::LINES)),
                    dim3(DP::RT), 0, s, in, out, nrows, tw, scale, (unsigned*)nullptr, 0, (float2*)nullptr);
}

// the rows of the data planes; *n_wsum (not null): the block sums of |W|^2 per frequency too
template <typename R, int N, typename TI, int T>
cudaError_t data_rows_launch(const TI* in, cx<R>* out, const Problem& P, const cx<R>* tw, unsigned* clear,
                             float2* wsum, int* n_wsum, cudaStream_t s) {
  using DP = DensePass<R, N, T>;
  const long long nrows = (long long)P.m1 * N;
  const dim3 g((unsigned)((nrows + DP::LINES - 1) / DP::LINES), P.n_omega);
  if constexpr (sizeof(R) == 4) {
    if (n_wsum) {
      *n_wsum = (int)g.x;
      return launch_pdl(k_fft_rows<R, N, false, TI, T, false, true>, g, dim3(DP::RT), 0, s, in, out, nrows, tw, R(1),
                        clear, clear_words(P), wsum);
    }
  }
  return launch_pdl(k_fft_rows<R, N, false, TI, T, false>, g, dim3(DP::RT), 0, s, in, out, nrows, tw, R(1), clear,
                    clear_words(P), (float2*)nullptr);
}

template <typename R, int N, bool INV, int T, bool D32>
cudaError_t cols_launch(const cx<R>* in, cx<R>* out, long long planes, const cx<R>* tw, cudaStream_t s) {
  using DP = DensePass<R, N, T>;
  constexpr long long MAX_Y = 32768;  // planes per launch (grid y <= 65535)
  for (long long p0 = 0; p0 < planes; p0 += MAX_Y) {
    const long long np = planes - p0 < MAX_Y ? planes - p0 : MAX_Y;
    const cudaError_t e = launch_pdl(k_fft_cols<R, N, INV, T, D32>, dim3((N + DP::COLS - 1) / DP::COLS, (unsigned)np),
                                     dim3(DP::CT), 0, s, in + p0 * N * N, out + p0 * N * N, tw);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// W (complex64) -> W~ (complex128 in w.wt64) and the norms: the forward transform
// of the mixed truncated-SVD route, in FP64
template <int N>
cudaError_t fwd_wide_impl(const float2* W, const Problem& P, const Work<float>& w, cudaStream_t s, cudaEvent_t mid) {
  const long long planes = (long long)P.n_omega * P.m1;
  cudaError_t e = data_rows_launch<double, N, float2, 0>(W, w.wt64, P, w.tw64, w.bar, nullptr, nullptr, s);
  if (e != cudaSuccess) return e;
  if (mid) cudaEventRecord(mid, s);
  e = cols_launch<double, N, false, 0, false>(w.wt64, w.wt64, planes, w.tw64, s);
  if (e != cudaSuccess) return e;
  const dim3 gn((unsigned)w.n_partial, (unsigned)P.n_omega);
  e = launch_pdl(k_mode_norms<double>, gn, dim3(NORM_T), 0, s, (const double2*)w.wt64, w.norms, w.partial, P.m1,
                 N * N, w.ctr);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

template <typename R, int N, int T>
cudaError_t fwd_tiled(const cx<R>* W, const Problem& P, const Work<R>& w, cudaStream_t s, cudaEvent_t mid,
                      bool norms, int* n_wsum, int* groups) {
  const bool early = norms && classify_early(P, sizeof(R) == 8);
  const cx<R>* tw = (const cx<R>*)w.tw;
  cudaError_t e = data_rows_launch<R, N, cx<R>, T>(W, w.wt, P, tw, w.bar, w.wsum, early ? n_wsum : nullptr, s);
  if (e != cudaSuccess) return e;
  if (mid) cudaEventRecord(mid, s);
  if constexpr (sizeof(R) == 4) {
    if (const int G = early ? norm_groups(P, false) : 0) {
      // columns and norms in one pass (the group sums in the profiles' place, still unused)
      using DP = DensePass<R, N, T>;
      const int ppg = (P.m1 + G - 1) / G;
      const dim3 g((N + DP::COLS - 1) / DP::COLS, (P.m1 + ppg - 1) / ppg, P.n_omega);
      *groups = (int)g.y;
      return launch_pdl(k_fft_cols_norms<R, N, T>, g, dim3(DP::CT), 0, s, (const cx<R>*)w.wt,
                        reinterpret_cast<R*>(w.prof), P.m1, ppg, tw);
    }
  }
  e = cols_launch<R, N, false, T, false>(w.wt, w.wt, (long long)P.n_omega * P.m1, tw, s);
  if (e != cudaSuccess) return e;
  if (early || !norms) return cudaGetLastError();
  return launch_mode_norms<R>(P, w, s);
}

template <int N>
cudaError_t active_impl(const Problem& P, const Work<float>& w, cudaStream_t s) {
  using AP = ActivePass<float, N>;
  constexpr int NCH = (N + AP::GC - 1) / AP::GC;
  const dim3 g((P.m1 + AP::GL - 1) / AP::GL, P.n_omega, NCH < 8 ? NCH : 8);
  return launch_pdl(k_fft_cols_active<float, N>, g, dim3(AP::NT), 0, s, w.wt, P.m1, (const unsigned*)w.colmask, w.tw);
}

template <typename R, int N>
cudaError_t fwd_impl(const cx<R>* W, const Problem& P, const Work<R>& w, cudaStream_t s, cudaEvent_t mid,
                     bool norms, int* n_wsum, int* groups) {
  if constexpr (std::is_same<R, float>::value) {
    if (w.wt64) return fwd_wide_impl<N>(W, P, w, s, mid);
    // N = 192 and 256: the cluster's row tiles (77 / 134 KB per CTA) leave one or two
    // CTAs per SM, and the two passes are faster (measured at 256^2 x 64, 29 planes, 6
    // frequencies: 0.139 ms vs 0.122 ms)
    if constexpr (N <= 128) {
      if (P.forward_single) return fwd_plane<R, N>(W, P, w, s, mid, norms, n_wsum);
    }
  }
  return P.fft_tile == 1 ? fwd_tiled<R, N, 1>(W, P, w, s, mid, norms, n_wsum, groups)
                         : fwd_tiled<R, N, 0>(W, P, w, s, mid, norms, n_wsum, groups);
}

template <typename R, int N>
cudaError_t dense_impl(const cx<R>* in, cx<R>* out, long long planes, bool inverse, const cx<R>* tw, cudaStream_t s) {
  constexpr bool D32 = sizeof(R) == 4;
  cudaError_t e;
  if (!inverse) {
    if ((e = rows_launch<R, N, false, cx<R>, 0, D32>(in, out, planes * N, tw, R(1), s)) != cudaSuccess) return e;
    return cols_launch<R, N, false, 0, D32>(out, out, planes, tw, s);
  }
  if ((e = cols_launch<R, N, true, 0, D32>(in, out, planes, tw, s)) != cudaSuccess) return e;
  return rows_launch<R, N, true, cx<R>, 0, D32>(out, out, planes * N, tw, R(1.0 / ((double)N * N)), s);
}

template <typename R, int N>
cudaError_t jvp_rows_impl(const Problem& P, int nd, const cx<R>* dv, const cx<R>* du, const cx<R>* Vx, const cx<R>* ux,
                          const R* xis, R* dxi, const cx<R>* tw, cudaStream_t s) {
  using JP = JvpPass<R, N>;
  const long long nrows = (long long)P.m * N;
  return launch_pdl(k_jvp_rows<R, N>, dim3((unsigned)nd, (unsigned)((nrows + JP::LINES - 1) / JP::LINES)), dim3(JP::NT),
                    0, s, P, dv, du, Vx, ux, xis, dxi, tw);
}

// F[xi F^-1 ut] -> out, M planes
template <typename R, int N>
cudaError_t xi_impl(const cx<R>* ut, cx<R>* out, const R* xi, long long planes, const cx<R>* tw, cudaStream_t s) {
  using DP = DensePass<R, N, 0>;
  constexpr bool D32 = sizeof(R) == 4;
  cudaError_t e = cols_launch<R, N, true, 0, D32>(ut, out, planes, tw, s);
  if (e != cudaSuccess) return e;
  const long long nrows = planes * N;
  constexpr size_t smem = sizeof(cx<R>) * LayIdx<Lay::ROW, N, DP::LINES, DP::SKEW>::ELEMS;
  static SmemOptIn attr;
  if ((e = opt_in_smem(attr, (const void*)k_rows_xi<R, N>, smem)) != cudaSuccess) return e;
  e = launch_pdl(k_rows_xi<R, N>, dim3((unsigned)((nrows + DP::LINES - 1) / DP::LINES)), dim3(DP::RT), smem, s, out,
                 xi, nrows, tw, R(1.0 / ((double)N * N)));
  if (e != cudaSuccess) return e;
  return cols_launch<R, N, false, 0, D32>(out, out, planes, tw, s);
}

template <typename R, int N>
cudaError_t real_impl(const R* xi, cx<R>* out, int m, const cx<R>* tw, cudaStream_t s) {
  using DP = DensePass<R, N, 0>;
  const long long npairs = (long long)m * N / 2;
  // A plain launch: about three blocks per SM, bound by the FP64 pipe, and those started while the
  // predecessor drains crowd on the SMs it has left (FP64, 37 planes of 192^2 in a row of calls: the
  // rows 77 us and the columns that start behind them 58 us; 35 and 31 us so)
  k_fft_rows_real<R, N><<<(unsigned)((npairs + DP::LINES - 1) / DP::LINES), DP::RT, 0, s>>>(xi, out, npairs, tw);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int ncols = m * (N / 2 + 1);
  return launch_pdl(k_fft_cols_real<R, N>, dim3((ncols + DP::COLS - 1) / DP::COLS), dim3(DP::CT), 0, s, out, ncols, tw);
}

}  // namespace

bool fft_size_supported(int n) {
#define FL_CASE(K) if (n == K) return true;
  FL_SIZES(FL_CASE)
#undef FL_CASE
  return false;
}

template <typename R>
cudaError_t launch_mode_norms(const Problem& P, const Work<R>& w, cudaStream_t s) {
  const dim3 gn((unsigned)w.n_partial, (unsigned)P.n_omega);
  cudaError_t e = launch_pdl(k_mode_norms<R>, gn, dim3(NORM_T), 0, s, (const cx<R>*)w.wt, w.norms, w.partial, P.m1,
                             P.n * P.n, w.ctr);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}
template cudaError_t launch_mode_norms<double>(const Problem&, const Work<double>&, cudaStream_t);
template cudaError_t launch_mode_norms<float>(const Problem&, const Work<float>&, cudaStream_t);

// FP32 from 8 MB of data planes up, where the traffic saved is worth an extra launch, in the
// two-pass transform under the discrepancy rule (a given alpha makes every column active).
// About six blocks per SM, each a run of planes.
int norm_groups(const Problem& P, bool fp64) {
  const bool two_passes = P.n > 128 || !P.forward_single;
  if (fp64 || !two_passes || P.alpha_mode != 0 || P.classify_single || wide_route(P, fp64)) return 0;
  if (8.0 * P.n_omega * P.m1 * P.n * P.n < 8e6) return 0;
  const int tiles = (P.n + 15) / 16 * P.n_omega;
  int G = (6 * sm_count() + tiles - 1) / tiles;
  G = G < P.m1 ? G : P.m1;
  return G < 4 * P.m ? G : 4 * P.m;  // the group sums fit in the profiles' place
}

cudaError_t launch_fft2_active(const Problem& P, const Work<float>& w, cudaStream_t s) {
  switch (P.n) {
#define FL_CASE(K) case K: return active_impl<K>(P, w, s);
    FL_SIZES(FL_CASE)
#undef FL_CASE
    default: return cudaErrorInvalidValue;
  }
}

template <typename R>
cudaError_t launch_fft2_forward(const cx<R>* W, const Problem& P, const Work<R>& w, cudaStream_t s,
                                cudaEvent_t mid, bool norms, int* n_wsum, int* groups) {
  switch (P.n) {
#define FL_CASE(K) case K: return fwd_impl<R, K>(W, P, w, s, mid, norms, n_wsum, groups);
    FL_SIZES(FL_CASE)
#undef FL_CASE
    default: return cudaErrorInvalidValue;
  }
}

template <typename R>
cudaError_t launch_fft2_dense(const cx<R>* in, cx<R>* out, int n, long long planes, bool inverse, const cx<R>* tw,
                              cudaStream_t s) {
  switch (n) {
#define FL_CASE(K) case K: return dense_impl<R, K>(in, out, planes, inverse, tw, s);
    FL_SIZES(FL_CASE)
#undef FL_CASE
    default: return cudaErrorInvalidValue;
  }
}
template cudaError_t launch_fft2_dense<double>(const double2*, double2*, int, long long, bool, const double2*, cudaStream_t);
template cudaError_t launch_fft2_dense<float>(const float2*, float2*, int, long long, bool, const float2*, cudaStream_t);

template <typename R>
cudaError_t launch_ifft_cols(const cx<R>* in, cx<R>* out, int n, long long planes, const cx<R>* tw, cudaStream_t s) {
  switch (n) {
#define FL_CASE(K) case K: return cols_launch<R, K, true, 0, sizeof(R) == 4>(in, out, planes, tw, s);
    FL_SIZES(FL_CASE)
#undef FL_CASE
    default: return cudaErrorInvalidValue;
  }
}
template cudaError_t launch_ifft_cols<double>(const double2*, double2*, int, long long, const double2*, cudaStream_t);
template cudaError_t launch_ifft_cols<float>(const float2*, float2*, int, long long, const float2*, cudaStream_t);

template <typename R>
cudaError_t launch_diff_jvp_rows(const Problem& P, int nd, const cx<R>* dv, const cx<R>* du, const cx<R>* Vx,
                                 const cx<R>* ux, const R* xis, R* dxi, const cx<R>* tw, cudaStream_t s) {
  switch (P.n) {
#define FL_CASE(K) case K: return jvp_rows_impl<R, K>(P, nd, dv, du, Vx, ux, xis, dxi, tw, s);
    FL_SIZES(FL_CASE)
#undef FL_CASE
    default: return cudaErrorInvalidValue;
  }
}
template cudaError_t launch_diff_jvp_rows<double>(const Problem&, int, const double2*, const double2*, const double2*,
                                                  const double2*, const double*, double*, const double2*,
                                                  cudaStream_t);
template cudaError_t launch_diff_jvp_rows<float>(const Problem&, int, const float2*, const float2*, const float2*,
                                                 const float2*, const float*, float*, const float2*, cudaStream_t);

template <typename R>
cudaError_t launch_xi_transform(const cx<R>* ut, cx<R>* out, const R* xi, int n, long long planes, const cx<R>* tw,
                                cudaStream_t s) {
  switch (n) {
#define FL_CASE(K) case K: return xi_impl<R, K>(ut, out, xi, planes, tw, s);
    FL_SIZES(FL_CASE)
#undef FL_CASE
    default: return cudaErrorInvalidValue;
  }
}
template cudaError_t launch_xi_transform<double>(const double2*, double2*, const double*, int, long long,
                                                 const double2*, cudaStream_t);
template cudaError_t launch_xi_transform<float>(const float2*, float2*, const float*, int, long long, const float2*,
                                                cudaStream_t);

template <typename R>
cudaError_t launch_fft2_real(const R* xi, cx<R>* out, int n, int m, const cx<R>* tw, cudaStream_t s) {
  switch (n) {
#define FL_CASE(K) case K: return real_impl<R, K>(xi, out, m, tw, s);
    FL_SIZES(FL_CASE)
#undef FL_CASE
    default: return cudaErrorInvalidValue;
  }
}
template cudaError_t launch_fft2_real<double>(const double*, double2*, int, int, const double2*, cudaStream_t);
template cudaError_t launch_fft2_real<float>(const float*, float2*, int, int, const float2*, cudaStream_t);

template <typename R>
cudaError_t launch_twiddles(cx<R>* tw, int n, cudaStream_t s) {
  k_twiddles<R><<<(n + 255) / 256, 256, 0, s>>>(tw, n);
  return cudaGetLastError();
}

template cudaError_t launch_fft2_forward<double>(const double2*, const Problem&, const Work<double>&, cudaStream_t,
                                                 cudaEvent_t, bool, int*, int*);
template cudaError_t launch_fft2_forward<float>(const float2*, const Problem&, const Work<float>&, cudaStream_t,
                                                cudaEvent_t, bool, int*, int*);
template cudaError_t launch_twiddles<double>(double2*, int, cudaStream_t);
template cudaError_t launch_twiddles<float>(float2*, int, cudaStream_t);

}  // namespace fl
