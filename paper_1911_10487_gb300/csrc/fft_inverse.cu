// Inverse 2D FFT passes of Algorithm 2 (step 2) with the pointwise recovery of step
// 3 fused into the last, for N = 2^a 3^b <= 256, in FP64 (double2) or FP32 (float2).
//
//   recover       : V~, U~ -> V = F^-1[V~], u = F^-1[U~] (Algorithm 2 step 2) and
//                   xi = Re(sum conj(u) V)/sum |u|^2, c = (c0^-2 - xi)^-1/2
//                   (step 3, Sec. 5.2; Sec. 1 for c).  The inverse column pass
//                   gathers the solved profiles of the active modes only and
//                   transforms only the columns nu1 that hold a nonzero mode; the
//                   row pass reads those columns by their positions and transforms
//                   full rows.
#include "fft_pass.cuh"

namespace fl {

namespace {

// ---- inverse pass 1: gather active profiles, columns (along y) ----------------
// A tile is GC columns of the compact column list by GL planes: the profiles lie plane-fastest
// per mode, so the GL planes of a mode are one 32-byte sector of the loads, and the GC columns
// one of the stores (16 columns of one plane before: a quarter of each sector used, and with 17
// active columns a second tile for one of them).  256^2 x 64, 8 frequencies, 137 columns: 27 us
// -> 21 us.
template <typename R, int N, int T> struct GatherPass {
  static constexpr bool F32 = sizeof(R) == 4;
  static constexpr int GC = 4, GL = (F32 ? 4 : 2) / (T == 0 ? 1 : 2), LINES = GC * GL;
  using PL = IoPlan<N, T == 0 ? 16 : 8, false>;
  static constexpr int NT = round32(LINES * N / (T == 0 ? (N % 3 == 0 ? 12 : 16) : 8)) < 256
                                ? round32(LINES * N / (T == 0 ? (N % 3 == 0 ? 12 : 16) : 8)) : 256;
};
constexpr int GATHER_COLS = 32;  // active columns the gather's grid covers in one pass (see rec_tiled)

// Element i of line b of a gather tile: column cb + b / GL, plane l0 + b % GL (the lanes
// of the loads go through the planes of a mode, those of the stores through both).  pre: the
// mode's slot (-1: zero), so that a thread's slot loads, then its profile loads, are in flight
// together.
template <typename R, int N, int GL> struct GatherLoad {
  const int* cols;      // of this frequency, from column cb on
  const int* slot;
  const cx<R>* prof;    // of this frequency, field and plane l0
  int nc, nl, stride;   // columns and planes of the tile, 2 M
  const cx<R>* inc;     // U~0 at nu = 0 on the tile's planes when that mode is inactive (else null)
  __device__ __forceinline__ int pre(int b, int i) const {
    return b / GL < nc && b % GL < nl ? slot[i * N + cols[b / GL]] : -1;
  }
  __device__ __forceinline__ cx<R> operator()(int b, int i, int s) const {
    if (s >= 0) return prof[(long long)s * stride + b % GL];
    return inc && i == 0 && b / GL == 0 ? inc[b % GL] : czero<R>();
  }
};

// Column chunks blockIdx.z, blockIdx.z + gridDim.z, ... of the compact column list of
// frequency om (grid below); field f = 0 (V~) or 1 (U~).  Inactive modes are zero in
// V~ and equal the incident field U~0 in U~; the plane wave exp(-i k0 z) has
// U~0 = N^2 exp(-i k0 z'_l) at nu = 0 and zero elsewhere.
template <typename R, int N, int T>
__global__ void __launch_bounds__((GatherPass<R, N, T>::NT))
k_ifft_cols_gather(Problem P, const cx<R>* __restrict__ prof, const int* __restrict__ slot,
                   const int* __restrict__ cols, const int* __restrict__ ncol,
                   cx<R>* __restrict__ t2, const cx<R>* __restrict__ tw) {
  using GP = GatherPass<R, N, T>;
  using PL = typename GP::PL;
  constexpr int GC = GP::GC, GL = GP::GL;
  __shared__ cx<R> buf[PL::stages > 1 ? N * GP::LINES : 1];
  __shared__ cx<R> tws[PL::tw_elems];
  __shared__ cx<R> inc[GL];
  load_stage_twiddles<R, PL, N, GP::NT>(tws, tw);  // a constant table: read while the predecessor drains
  pdl_wait();
  pdl_trigger();
  // grid (ceil(M / GL), 2 n_omega, chunks): the column chunk is the slowest index, so that
  // the chunks that hold active columns are dispatched first and the rest, which return at
  // once, last; a block loops when ncol needs more chunks
  const int om = blockIdx.y >> 1, f = blockIdx.y & 1;
  const int l0 = blockIdx.x * GL;
  const int nc = ncol[om];
  const long long N2 = (long long)N * N;
  const int M = P.m;
  const int* sl = slot + om * N2;
  const cx<R>* pr = prof + (long long)om * N2 * 2 * M + f * M + l0;
  cx<R>* dst = t2 + ((long long)om * 2 + f) * M * N2 + l0 * N2;
  for (int cb = blockIdx.z * GC; cb < nc; cb += gridDim.z * GC) {
    // column 0 of the list is nu1 = 0 (it always holds the incident mode)
    const bool wave = cb == 0 && f == 1 && !P.incident && sl[0] < 0;
    if (wave && threadIdx.x < GL) {
      double sn, cs;
      sincos(-(P.omega[om] / P.c0) * (P.z1 + (l0 + threadIdx.x + 0.5) * P.hz), &sn, &cs);
      inc[threadIdx.x] = from_d<R>(make_double2((double)N2 * cs, (double)N2 * sn));
    }
    if (wave || cb != (int)blockIdx.z * GC) __syncthreads();  // (the previous chunk's last stage has read buf)
    const int ncb = min(GC, nc - cb), nlb = min(GL, M - l0);
    fft_lines_io<R, PL, N, true, GP::LINES, GP::NT, Lay::COL, 0, true>(
        buf, tws, GatherLoad<R, N, GL>{cols + om * N + cb, sl, pr, ncb, nlb, 2 * M, wave ? inc : nullptr},
        [&](int b, int i, cx<R> v) {
          if (b / GL < ncb && b % GL < nlb) dst[(b % GL) * N2 + i * N + cb + b / GL] = v;
        });
  }
}

template <int NT> __device__ __forceinline__ unsigned long long block_sum_u64(unsigned v, unsigned* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  unsigned long long s = 0;
  if (threadIdx.x == 0)
    for (int w = 0; w < NT / 32; ++w) s += red[w];
  return s;
}

// ---- inverse pass 2: rows (along x) + step 3 ----------------------------------
// a / b and 1/sqrt(x) of the pointwise recovery: IEEE in FP32; in FP64 by
// Newton-Raphson from FP32 seeds (rcp64, rsqrt64), a few dependent FP64 operations
// instead of the FP64 division and square root, which dominate this kernel on a
// GPU whose FP64 pipe runs at 1/64 of the FP32 rate.
template <typename R> __device__ __forceinline__ R quot(R a, R b);
template <> __device__ __forceinline__ float quot<float>(float a, float b) { return a / b; }
template <> __device__ __forceinline__ double quot<double>(double a, double b) { return a * rcp64(b); }
template <typename R> __device__ __forceinline__ R inv_sqrt(R x);
template <> __device__ __forceinline__ float inv_sqrt<float>(float x) { return rsqrtf(x); }  // <= 2 ulp
template <> __device__ __forceinline__ double inv_sqrt<double>(double x) { return rsqrt64(x); }

// xi and c of the PER elements of the thread from the least-squares sums, and the counters of
// guarded, NaN-c and non-finite voxels (almost always zero, so one barrier decides).  at(p):
// offset of element p in xi, negative for none.  guard: the least den of a kept voxel
// (host-derived: no FP64 division on the device)
template <typename R, int PER, int NT, class At>
__device__ __forceinline__ void recover_epilogue(const Problem& P, const R* num, const R* den, R guard, At at,
                                                 R* __restrict__ xi, R* __restrict__ cout,
                                                 unsigned long long* __restrict__ ctr, unsigned* red) {
  const R inv_c02 = sizeof(R) == 4 ? R(P.inv_c02_f) : R(P.inv_c02);
  unsigned n_guard = 0, n_nan = 0, n_bad = 0;
#pragma unroll
  for (int p = 0; p < PER; ++p) {
    const long long o = at(p);
    if (o >= 0) {
      const bool g = !(den[p] >= guard);
      const R x = g ? R(0) : quot<R>(num[p], den[p]);
      n_guard += g;
      n_bad += !isfinite(x);
      xi[o] = x;
      if (cout) {
        const bool ok = x < inv_c02;
        n_nan += !ok;
        cout[o] = ok ? inv_sqrt<R>(inv_c02 - x) : R(NAN);
      }
    }
  }
  if (__syncthreads_or((n_guard | n_nan | n_bad) != 0u)) {
    const unsigned long long sg = block_sum_u64<NT>(n_guard, red);
    __syncthreads();
    const unsigned long long sn = block_sum_u64<NT>(n_nan, red);
    __syncthreads();
    const unsigned long long sb = block_sum_u64<NT>(n_bad, red);
    if (threadIdx.x == 0) {
      if (sg) atomicAdd(ctr + C_U_GUARD, sg);
      if (sn) atomicAdd(ctr + C_NAN_C, sn);
      if (sb) atomicAdd(ctr + C_NONFINITE, sb);
    }
  }
}

// The recovery pass: LINES rows of X per block, their V and u lines together (lines 0 .. LINES
// - 1 and LINES .. 2 LINES - 1 of the tile).  The compact columns of the next frequency are
// staged by asynchronous copies while this one is transformed; the first stage reads them
// through the position of each column in the list, leaving out the inputs of columns that the
// list's band does not reach; the last stage goes back over its own inputs in the tile, and each
// thread then adds its voxels' V and u to the least-squares sums in registers.
// What bounds it: shared memory and latency in FP32, the FP64 pipe in FP64.  Clearing the tile,
// scattering the columns and every stage in place took six crossings of shared memory and five
// barriers per frequency: 256^2 x 64, 8 frequencies (FP32) 171 us; this split without staging
// and band 146 us, with both 117 us (100 us as pairs, RecPair); 128^2 x 71, 3 frequencies, incident field (FP64) 435 us ->
// 322 us, 256 us of it FP64 instructions.  (A V and a u butterfly held in registers beside the
// sums, one crossing fewer, left half the resident blocks: 131 us.)
// The sums are taken of the unscaled transforms (raw: N^2 V and N^2 u, a given incident field
// times N^2) in FP64: xi is their quotient either way, and the guard on sum |u|^2 is scaled
// instead (Problem::u_guard_raw), which saves FP64 products per voxel and frequency.
template <typename R, int N, int T> struct RecPass {
  static constexpr bool F32 = sizeof(R) == 4;
  // Radices that give each stage of a small FP64 tile whole warps, against 16 throughout: one
  // frequency, 16 planes: N = 16 16.3 us (20.1), 32 19.3 (23.2), 64 45.1 (45.1); 4 frequencies, 64 planes:
  // 32 95 (103), but 16 68 (55) and 64 194 (157), where the tiles fill the chip and fewer stages win
  static constexpr int MAXR = T == 1 ? 8 : F32 ? 16 : (N == 16 ? 4 : N <= 64 ? 8 : 16);
  using PL = IoPlan<N, MAXR, false>;
  static constexpr int NT = F32 ? (N >= 192 ? 256 : 128) : (N >= 192 ? 128 : 64);
  static constexpr int ROWS0 = F32 ? (N <= 16 ? 16 : 8) : (N <= 16 ? 8 : 4);
  static constexpr int LINES = T == 0 ? (F32 && N == 256 ? 4 : ROWS0) : ROWS0 / 2;
  static constexpr int SKEW = 16;
  // resident blocks the registers are held to: at 128^2 x 64 the pass's 1024 blocks at once (72
  // registers, 52-64 bytes of them spilled at N = 128).  128^2 x 64, 4 frequencies: 24.3 us, 27.4
  // without; 128^2 x 16, one frequency: 7.5 and 7.0.  N = 64: the same registers either way; the other
  // lengths lose by it (96^2 x 64, 4 frequencies: 20.9 us as here, 25.1 held to 7)
  static constexpr int MINB = !F32 || T == 1 ? 1 : N >= 192 ? 3 : (N == 128 || N == 64) ? 7 : 1;
  static constexpr int SC = !F32 && N == 256 ? 16 : 32;  // staged columns per row (RecStage)
  static constexpr int E = LINES * N, PER = (E + NT - 1) / NT;  // voxels of the block, of a thread
  using IX = LayIdx<Lay::ROW, N, 2 * LINES, SKEW>;
};

// Lengths from which V and u run as packed pairs (RecPair): a thread holds twice the registers, so half
// the warps; below, the pass is one wave of short blocks bound by latency (128^2 x 64: 11 us, 14 us
// as pairs; the whole dense step 60 -> 64 us).
constexpr int PAIR_N = 192;

template <typename R> __host__ __device__ constexpr bool raw_sums() { return sizeof(R) == 8; }

// What a block stages of the next frequency while it transforms this one: the columns of its
// rows (at most RecPass::SC; more are read from global memory by the first stage) and the positions of
// the columns in the list.
template <typename R, int N, int T> struct RecStage {
  cx<R> col[2][2 * RecPass<R, N, T>::LINES][RecPass<R, N, T>::SC];
  int pos[2][N];
};

// The first stage of a radix-16 plan when only the first and the last E sixteenths of the columns
// hold anything (low wavenumbers; E = 8: no such bound): butterfly j has inputs j + r N/16.
template <typename R, int N, int T, int E, class Ld>
__device__ __forceinline__ void recover_first(cx<R>* buf, Ld ld) {
  using RP = RecPass<R, N, T>;
  constexpr int NB = N / 16, TOTAL = 2 * RP::LINES * NB;
  for (int t = threadIdx.x; t < TOTAL; t += RP::NT) {
    const int b = t / NB, j = t % NB;
    cx<R> v[16];
#pragma unroll
    for (int r = 0; r < 16; ++r)
      if (r < E || r >= 16 - E) v[r] = ld(b, j + r * NB);
    if constexpr (E == 8) Dft<R, true>::d16(v);
    else Dft<R, true>::template d16_edge<E>(v);
#pragma unroll
    for (int r = 0; r < 16; ++r) buf[RP::IX::at(b, j * 16 + r)] = v[r];
  }
}

// FP32, two stages, T = 0: V and u of a voxel as one packed pair (pair.cuh).  Both fields take the
// same butterflies with the same twiddles, so every operation is one packed instruction, a twiddle is
// read once for both, and the sums come straight from the last stage's registers (recover_pass takes
// them through the tile, one more write and read).  256^2 x 64, 8 frequencies: 117 us -> 100 us, the
// batch of 32 smaller problems 1.37 -> 1.32 ms; bound by issue slots and latency at 16 warps per SM
// (54% of the slots; 128 registers, of which the FP64 redo and the sums spill 192 bytes at N = 256, 360
// with a given incident field, and 16-48 at 192; a tile of 4 rows at N = 256: static shared memory holds
// no 8).
template <typename R, int N, int T> struct RecPair {
  using RP = RecPass<R, N, T>;
  using PL = typename RP::PL;
  static constexpr bool use = sizeof(R) == 4 && T == 0 && PL::stages == 2 && N >= PAIR_N;
  static constexpr int LINES = RP::LINES, R0 = PL::radix(0), R1 = PL::radix(1), NB = N / R1;
  static constexpr int NT = LINES * NB < 128 ? LINES * NB : 128;  // one last-stage butterfly per thread
  static constexpr int PERB = (LINES * NB + NT - 1) / NT, PER = PERB * R1;
  using IX = LayIdx<Lay::ROW, N, LINES, RP::SKEW>;
};

// recover_pass on packed pairs: the voxel of sum p is (line, element) = RecPair's last-stage outputs
template <int N, typename A, bool INC>
__device__ __forceinline__ void recover_pass_pairs(const Problem& P, const float2* __restrict__ t2,
                                                   const int* __restrict__ colpos, const int* __restrict__ ncol,
                                                   const int* __restrict__ colseg, const float2* __restrict__ u0,
                                                   cf2* buf, const cf2* tws, RecStage<float, N, 0>& stg, A* num,
                                                   A* den) {
  using RP = RecPass<float, N, 0>;
  using PR = RecPair<float, N, 0>;
  using IX = typename PR::IX;
  constexpr int LINES = PR::LINES, NT = PR::NT, SC = RP::SC, R0 = PR::R0, R1 = PR::R1, NB0 = N / R0, NB = PR::NB;
  const long long nrows = (long long)P.m * N;
  const long long row0 = (long long)blockIdx.x * LINES;
  const int rows = (int)(nrows - row0 < LINES ? nrows - row0 : LINES);
  const long long uoff = nrows * N;  // u behind V by nrows rows
  const f2 scale = f2(P.inv_n2_f);
#pragma unroll
  for (int p = 0; p < PR::PER; ++p) { num[p] = A(0); den[p] = A(0); }
  auto stage = [&](int om, int nc) {
    const float2* src = t2 + ((long long)om * 2 * nrows + row0) * N;
    if (nc <= SC)
      for (int q = threadIdx.x; q < 2 * LINES * SC; q += NT) {
        const int line = q / SC, c = q % SC, bl = line >= LINES ? line - LINES : line;
        if (c < nc && bl < rows)
          async_copy(&stg.col[om & 1][line][c], (line >= LINES ? src + uoff : src) + bl * N + c);
      }
    for (int i = threadIdx.x; i < N; i += NT) async_copy(&stg.pos[om & 1][i], colpos + om * N + i);
  };
  int nc = ncol[0];
  stage(0, nc);
  for (int om = 0; om < P.n_omega; ++om) {
    const int seg = colseg[om];
    const int nc1 = om + 1 < P.n_omega ? ncol[om + 1] : 0;
    async_wait();
    __syncthreads();  // this frequency's columns are staged, and the tile has been read
    if (om + 1 < P.n_omega) stage(om + 1, nc1);
    const int* ps = stg.pos[om & 1];
    const float2* src = t2 + ((long long)om * 2 * nrows + row0) * N;
    const bool staged = nc <= SC;
    auto ld = [&](int b, int i) {
      const int c = ps[i];
      if (c < 0 || b >= rows) return cf2{f2(0.f), f2(0.f)};
      return staged ? pair_of(stg.col[om & 1][b][c], stg.col[om & 1][LINES + b][c])
                    : pair_of(src[b * N + c], src[uoff + b * N + c]);
    };
    auto first = [&](auto edge) {
      constexpr int E = decltype(edge)::value;
      for (int t = threadIdx.x; t < LINES * NB0; t += NT) {
        const int b = t / NB0, j = t % NB0;
        cf2 v[R0];
#pragma unroll
        for (int r = 0; r < R0; ++r)
          if (E == 0 || r < E || r >= R0 - E) v[r] = ld(b, j + r * NB0);
        if constexpr (E == 0) Dft<f2, true>::template run<R0>(v);
        else Dft<f2, true>::template d16_edge<E>(v);
#pragma unroll
        for (int r = 0; r < R0; ++r) buf[IX::at(b, j * R0 + r)] = v[r];
      }
    };
    if constexpr (R0 == 16) {
      if ((seg & ~0x8001) == 0) first(std::integral_constant<int, 1>());
      else if ((seg & ~0xC003) == 0) first(std::integral_constant<int, 2>());
      else first(std::integral_constant<int, 0>());
    } else {
      first(std::integral_constant<int, 0>());
    }
    __syncthreads();
#pragma unroll
    for (int pb = 0; pb < PR::PERB; ++pb) {
      const int t = threadIdx.x + pb * NT;
      if ((LINES * NB) % NT == 0 || t < LINES * NB) {
        const int b = t / NB, j = t % NB;
        cf2 v[R1];
        io_butterfly<f2, typename RP::PL, N, true, LINES, Lay::ROW, RP::SKEW, 1>(buf, tws, b, j, v);
#pragma unroll
        for (int r = 0; r < R1; ++r) {
          const float2 re = (scale * v[r].x).split(), im = (scale * v[r].y).split();  // (V, u)
          float2 u = make_float2(re.y, im.y);
          if (INC && b < rows) u = u + u0[((long long)om * nrows + row0 + b) * N + j + r * NB];  // U~ - U~0
          num[pb * R1 + r] += (A)u.x * (A)re.x + (A)u.y * (A)im.x;  // Re(conj(u) V)
          den[pb * R1 + r] += (A)u.x * (A)u.x + (A)u.y * (A)u.y;    // |u|^2
        }
      }
    }
    nc = nc1;
  }
  __syncthreads();  // (a second pass reuses the tile and the staged columns)
}

// the sums of the thread's voxels e = threadIdx.x + p NT over the frequencies, in the
// accumulator type A
template <typename R, int N, typename A, bool INC, int T>
__device__ __forceinline__ void recover_pass(const Problem& P, const cx<R>* __restrict__ t2,
                                             const int* __restrict__ colpos, const int* __restrict__ ncol,
                                             const int* __restrict__ colseg, const cx<R>* __restrict__ u0, cx<R>* buf,
                                             const cx<R>* tws, RecStage<R, N, T>& stg, A* num, A* den) {
  using RP = RecPass<R, N, T>;
  using PL = typename RP::PL;
  using IX = typename RP::IX;
  constexpr int LINES = RP::LINES, NT = RP::NT, E = RP::E, PER = RP::PER, SC = RP::SC;
  const long long nrows = (long long)P.m * N;
  const long long row0 = (long long)blockIdx.x * LINES;
  const int rows = (int)(nrows - row0 < LINES ? nrows - row0 : LINES);
  const long long uoff = nrows * N;  // u behind V by nrows rows
  const R scale = sizeof(R) == 4 ? R(P.inv_n2_f) : R(P.inv_n2);
  const R n2 = R((double)N * N);
#pragma unroll
  for (int p = 0; p < PER; ++p) { num[p] = A(0); den[p] = A(0); }
  auto stage = [&](int om, int nc) {
    const cx<R>* src = t2 + ((long long)om * 2 * nrows + row0) * N;
    if (nc <= SC)
      for (int q = threadIdx.x; q < 2 * LINES * SC; q += NT) {
        const int line = q / SC, c = q % SC, bl = line >= LINES ? line - LINES : line;
        if (c < nc && bl < rows)
          async_copy(&stg.col[om & 1][line][c], (line >= LINES ? src + uoff : src) + bl * N + c);
      }
    for (int i = threadIdx.x; i < N; i += NT) async_copy(&stg.pos[om & 1][i], colpos + om * N + i);
  };
  int nc = ncol[0];
  stage(0, nc);
  for (int om = 0; om < P.n_omega; ++om) {
    const int seg = colseg[om];
    const int nc1 = om + 1 < P.n_omega ? ncol[om + 1] : 0;
    async_wait();
    __syncthreads();  // this frequency's columns are staged, and the tile has been read
    if (om + 1 < P.n_omega) stage(om + 1, nc1);
    const int* ps = stg.pos[om & 1];
    const cx<R>* src = t2 + ((long long)om * 2 * nrows + row0) * N;
    const bool staged = nc <= SC;
    auto ld = [&](int line, int i) {
      const int c = ps[i], bl = line >= LINES ? line - LINES : line;
      if (c < 0 || bl >= rows) return czero<R>();
      return staged ? stg.col[om & 1][line][c] : (line >= LINES ? src + uoff : src)[bl * N + c];
    };
    auto st = [&](int line, int i, cx<R> v) { buf[IX::at(line, i)] = v; };
    if constexpr (PL::stages == 2 && PL::radix(0) == 16) {
      if ((seg & ~0x8001) == 0) recover_first<R, N, T, 1>(buf, ld);
      else if ((seg & ~0xC003) == 0) recover_first<R, N, T, 2>(buf, ld);
      else recover_first<R, N, T, 8>(buf, ld);
      __syncthreads();
      io_last<R, PL, N, true, 2 * LINES, NT, Lay::ROW, RP::SKEW>(buf, tws, st);
    } else {
      fft_lines_io<R, PL, N, true, 2 * LINES, NT, Lay::ROW, RP::SKEW>(buf, tws, ld, st);
    }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      const int e = threadIdx.x + p * NT;
      if (E % NT == 0 || e < E) {
        const int b = e / N, i = e % N;
        cx<R> v = buf[IX::at(b, i)], u = buf[IX::at(LINES + b, i)];
        if constexpr (!raw_sums<R>()) {
          v = scale * v;
          u = scale * u;
        }
        if (INC && b < rows) {  // the transform holds U~ - U~0
          const cx<R> w = u0[((long long)om * nrows + row0) * N + e];
          if constexpr (raw_sums<R>()) u = mk<R>(fma(n2, w.x, u.x), fma(n2, w.y, u.y));
          else u = u + w;
        }
        num[p] += (A)u.x * (A)v.x + (A)u.y * (A)v.y;  // Re(conj(u) V)
        den[p] += (A)u.x * (A)u.x + (A)u.y * (A)u.y;  // |u|^2
      }
    }
    nc = nc1;
  }
  __syncthreads();  // (a second pass reuses the tile and the staged columns)
}

// Shape of the recovery kernel: threads, sums per thread, tile
template <typename R, int N, int T, bool P = RecPair<R, N, T>::use> struct RecForm {
  using RP = RecPass<R, N, T>;
  using V = R;
  using IX = typename RP::IX;
  static constexpr bool PAIRS = false;
  static constexpr int NT = RP::NT, PER = RP::PER, MINB = RP::MINB;
};
template <typename R, int N, int T> struct RecForm<R, N, T, true> {
  using PR = RecPair<R, N, T>;
  using V = f2;
  using IX = typename PR::IX;
  static constexpr bool PAIRS = true;
  static constexpr int NT = PR::NT, PER = PR::PER, MINB = 512 / PR::NT;
};

// INC: u0 (the incident field on X) is given and added to u; otherwise the transform
// already holds the plane wave
template <typename R, int N, bool INC, int T>
__global__ void __launch_bounds__((RecForm<R, N, T>::NT), (RecForm<R, N, T>::MINB))
k_ifft_rows_recover(Problem P, const cx<R>* __restrict__ t2, const int* __restrict__ colpos,
                    const int* __restrict__ ncol, const int* __restrict__ colseg, const cx<R>* __restrict__ u0, R* __restrict__ xi, R* __restrict__ cout,
                    unsigned long long* __restrict__ ctr, const cx<R>* __restrict__ tw) {
  using RP = RecPass<R, N, T>;
  using PL = typename RP::PL;
  using RF = RecForm<R, N, T>;
  using C = cx<typename RF::V>;
  constexpr int NT = RF::NT, PER = RF::PER;
  __shared__ C buf[RF::IX::ELEMS];
  __shared__ C tws[PL::tw_elems];
  __shared__ RecStage<R, N, T> stg;
  __shared__ unsigned red[NT / 32];
  if constexpr (RF::PAIRS) load_stage_twiddles_pairs<PL, N, NT>(tws, tw);
  else load_stage_twiddles<R, PL, N, NT>(tws, tw);  // a constant table: read while the predecessor drains
  pdl_wait();
  pdl_trigger();
  const long long nrows = (long long)P.m * N;
  const long long row0 = (long long)blockIdx.x * RP::LINES;
  const int el = (int)(nrows - row0 < RP::LINES ? nrows - row0 : RP::LINES) * N;  // voxels of this block
  auto at = [&](int p) {  // the block's voxel of the thread's sum p (el or more: none)
    if constexpr (RF::PAIRS) {
      using PR = RecPair<R, N, T>;
      const int t = threadIdx.x + p / PR::R1 * NT;
      return t / PR::NB * N + t % PR::NB + p % PR::R1 * PR::NB;
    } else {
      return (int)threadIdx.x + p * NT;
    }
  };
  auto pass = [&](auto* n, auto* d) {
    using A = std::remove_pointer_t<decltype(n)>;
    if constexpr (RF::PAIRS)
      recover_pass_pairs<N, A, INC>(P, t2, colpos, ncol, colseg, u0, buf, tws, stg, n, d);
    else
      recover_pass<R, N, A, INC, T>(P, t2, colpos, ncol, colseg, u0, buf, tws, stg, n, d);
  };
  R num[PER], den[PER];
  const double gd = raw_sums<R>() ? P.u_guard_raw : P.u_guard;
  R guard = sizeof(R) == 4 ? R(P.u_guard_f) : R(gd);
  bool redo = sizeof(R) == 4 && P.sums64;
  if (!redo) {
    pass(num, den);
    if constexpr (sizeof(R) == 4) {
      bool bad = false;
#pragma unroll
      for (int p = 0; p < PER; ++p)
        bad |= at(p) < el && !(isfinite(num[p]) && isfinite(den[p]));
      redo = __syncthreads_or(bad) != 0;
    }
  }
  if constexpr (sizeof(R) == 4) {
    if (redo) {
      // the sums left the range of R (|u| |V| beyond FP32 for huge evanescent profiles), or
      // were asked for in FP64: FP64 sums; xi itself is in range
      double nd[PER], dd[PER];
      pass(nd, dd);
#pragma unroll
      for (int p = 0; p < PER; ++p) {
        const bool g = !(dd[p] >= gd);
        num[p] = g ? R(0) : R(nd[p] / dd[p]);
        den[p] = g ? R(0) : R(1);
      }
      guard = R(0.5);  // den is now 1 (kept) or 0 (guarded)
    }
  }
  recover_epilogue<R, PER, NT>(
      P, num, den, guard,
      [&](int p) {
        const int e = at(p);
        return e < el ? row0 * N + e : -1LL;
      },
      xi, cout, ctr, red);
}

// ---- single-pass inverse transform and recovery: one X plane per cluster ---------
// grid (C, M), clusters of C = plane_cluster<N>() CTAs along x; CTA r of the cluster
// of plane l owns rows r RB .. r RB + RB - 1 (RB = N / C) of both fields (V and u) in
// its shared memory.  For every frequency the cluster splits the 2 nc active columns
// (V~ and U~ columns nu1 of cols) among its CTAs; each gathers its columns' profiles
// (as k_ifft_cols_gather), transforms them along y and stores every value in the row
// tile of the CTA that owns its row (distributed shared memory).  After a cluster
// barrier each CTA transforms its rows along x and accumulates the least-squares sums
// (as recover_pass).  No intermediate array goes through global memory, and one launch
// replaces two.
constexpr int REC_CL = 8;  // column lines per chunk (a divisor of THREADS)

template <typename R, int N> __host__ __device__ constexpr size_t plane_rec_smem() {
  constexpr int RB = N / plane_cluster<N>();
  return sizeof(cx<R>) * ((size_t)LayIdx<Lay::ROW, N, 2 * RB, 8>::ELEMS + (size_t)REC_CL * N + N);
}

// The sums of the elements p0 .. p0 + G - 1 (of threadIdx.x + p THREADS < RB N) over
// the frequencies, in the accumulator type A.  Called by every thread of every CTA of
// the cluster (it holds cluster barriers).
template <typename R, int N, bool INC, typename A, int G>
__device__ __forceinline__ void plane_rec_pass(const Problem& P, const cx<R>* __restrict__ prof,
                                               const int* __restrict__ slot, const int* __restrict__ cols,
                                               const int* __restrict__ ncol, const cx<R>* __restrict__ u0, int l,
                                               unsigned r, cx<R>* rt, cx<R>* ct, const cx<R>* tw_s, int p0, A* num,
                                               A* den) {
  constexpr int C = plane_cluster<N>(), RB = N / C;
  using IX = LayIdx<Lay::ROW, N, 2 * RB, 8>;  // V rows, then u rows
  constexpr int E = RB * N;
  const int M = P.m;
  const long long N2 = (long long)N * N;
  const R scale = R(1.0 / (double)N2);
#pragma unroll
  for (int k = 0; k < G; ++k) { num[k] = A(0); den[k] = A(0); }
  for (int om = 0; om < P.n_omega; ++om) {
    for (int e = threadIdx.x; e < IX::ELEMS; e += THREADS) rt[e] = czero<R>();
    cluster_sync();  // every row tile is cleared (and was read) before any CTA stores into it
    const int nc = ncol[om];
    const int* cl = cols + om * N;
    const int nl = 2 * nc, lpc = (nl + C - 1) / C;  // line q: field q / nc, column cl[q % nc]
    const int q0 = min(nl, (int)r * lpc), q1 = min(nl, q0 + lpc);
    // thread t handles line b = t % REC_CL of each chunk, rows i = t / REC_CL + p THREADS / REC_CL:
    // one column per thread, its CPER values' loads issued together
    constexpr int CPER = (REC_CL * N + THREADS - 1) / THREADS;
    const int b = threadIdx.x % REC_CL;
    for (int c0 = q0; c0 < q1; c0 += REC_CL) {
      const int q = c0 + b;
      const int f = q >= nc ? 1 : 0;
      const int nu1 = q < q1 ? cl[q - f * nc] : -1;
      int sl[CPER];
#pragma unroll
      for (int p = 0; p < CPER; ++p) {
        const int i = threadIdx.x / REC_CL + p * (THREADS / REC_CL);
        sl[p] = (nu1 >= 0 && i < N) ? slot[om * N2 + (long long)i * N + nu1] : -1;
      }
#pragma unroll
      for (int p = 0; p < CPER; ++p) {
        const int i = threadIdx.x / REC_CL + p * (THREADS / REC_CL);
        if (i < N) {
          cx<R> v = czero<R>();
          if (sl[p] >= 0) {
            v = prof[(((long long)om * N2 + sl[p]) * 2 + f) * M + l];
          } else if (!INC && f == 1 && i == 0 && nu1 == 0) {
            // the plane wave's U~0 = N^2 exp(-i k0 z'_l) at nu = 0: the phase reduced to
            // [-pi, pi] in FP64, its sine and cosine in FP32 (the precision of R)
            const double ph = -(P.omega[om] / P.c0) * (P.z1 + (l + 0.5) * P.hz);
            const double red = fma(-6.283185307179586, rint(ph * 0.15915494309189535), ph);
            float sn, cs;
            sincosf((float)red, &sn, &cs);
            v = mk<R>(R(N2) * R(cs), R(N2) * R(sn));
          }
          ct[i * REC_CL + b] = v;  // element i of line b
        }
      }
      __syncthreads();
      fft_lines<R, N, true, REC_CL, THREADS, Lay::COL, 8>(ct, tw_s);
      if (nu1 >= 0) {  // value i of the line -> row i % RB of CTA i / RB
#pragma unroll
        for (int p = 0; p < CPER; ++p) {
          const int i = threadIdx.x / REC_CL + p * (THREADS / REC_CL);
          if (i < N) dsmem_st(dsmem_addr(rt + IX::at(f * RB + i % RB, nu1), (unsigned)(i / RB)), ct[i * REC_CL + b]);
        }
      }
      __syncthreads();
    }
    cluster_sync();  // every active column has reached its rows
    fft_lines<R, N, true, 2 * RB, THREADS, Lay::ROW, 8, 8>(rt, tw_s);
#pragma unroll
    for (int k = 0; k < G; ++k) {
      const int e = threadIdx.x + (p0 + k) * THREADS;
      if (e < E) {
        const cx<R> v = scale * rt[IX::at(e / N, e % N)];
        cx<R> u = scale * rt[IX::at(RB + e / N, e % N)];
        if (INC) u = u + u0[((long long)om * M + l) * N2 + (long long)((int)r * RB + e / N) * N + (e % N)];
        num[k] += (A)u.x * (A)v.x + (A)u.y * (A)v.y;  // Re(conj(u) V)
        den[k] += (A)u.x * (A)u.x + (A)u.y * (A)u.y;  // |u|^2
      }
    }
    __syncthreads();
  }
}

template <typename R, int N, bool INC>
__global__ void __launch_bounds__(THREADS, 2)
k_ifft2_plane_recover(Problem P, const cx<R>* __restrict__ prof, const int* __restrict__ slot,
                      const int* __restrict__ cols, const int* __restrict__ ncol, const cx<R>* __restrict__ u0,
                      R* __restrict__ xi, R* __restrict__ cout, unsigned long long* __restrict__ ctr,
                      const cx<R>* __restrict__ tw) {
  constexpr int C = plane_cluster<N>(), RB = N / C;
  constexpr int E = RB * N;
  constexpr int PER = (E + THREADS - 1) / THREADS;
  static_assert(PER <= 32, "one bit per element in the redo mask");
  constexpr int G = 2;  // elements per thread of one redo pass
  extern __shared__ __align__(16) unsigned char plane_smem[];
  cx<R>* rt = reinterpret_cast<cx<R>*>(plane_smem);
  cx<R>* ct = rt + LayIdx<Lay::ROW, N, 2 * RB, 8>::ELEMS;
  cx<R>* tw_s = ct + REC_CL * N;
  __shared__ unsigned red[THREADS / 32];
  __shared__ unsigned vote[8];
  load_twiddles<R, N>(tw_s, tw);  // a constant table: read while the predecessor drains
  pdl_wait();
  pdl_trigger();
  const unsigned r = cluster_rank();
  const int l = blockIdx.y;
  const long long row0 = (long long)l * N + (long long)r * RB;
  R num[PER], den[PER];
  unsigned any = 1;
  if (!P.sums64) {
    plane_rec_pass<R, N, INC, R, PER>(P, prof, slot, cols, ncol, u0, l, r, rt, ct, tw_s, 0, num, den);
    bool bad = false;
#pragma unroll
    for (int p = 0; p < PER; ++p) bad |= !(isfinite(num[p]) && isfinite(den[p]));
    const unsigned mine = __syncthreads_or(bad) ? 1u : 0u;
    // every CTA of the cluster learns whether any of them overflowed
    if (threadIdx.x < C) dsmem_st(dsmem_addr(&vote[r], threadIdx.x), mine);
    cluster_sync();
    any = 0;
#pragma unroll
    for (int q = 0; q < C; ++q) any |= vote[q];
  }
  if (any) {
    // the sums left the range of R (|u| |V| beyond FP32 for huge evanescent profiles):
    // the cluster redoes the plane with FP64 sums, G elements per thread at a time;
    // the quotient goes through xi (written and read back by the same thread)
    unsigned gated = 0;
    for (int p0 = 0; p0 < PER; p0 += G) {
      double nd[G], dd[G];
      plane_rec_pass<R, N, INC, double, G>(P, prof, slot, cols, ncol, u0, l, r, rt, ct, tw_s, p0, nd, dd);
#pragma unroll
      for (int k = 0; k < G; ++k) {
        const int e = threadIdx.x + (p0 + k) * THREADS;
        if (p0 + k < PER && e < E) {
          const bool g = !(dd[k] >= (double)P.n_omega * P.eps_u * P.eps_u);
          gated |= (g ? 1u : 0u) << (p0 + k);
          xi[(row0 + e / N) * N + (e % N)] = g ? R(0) : R(nd[k] / dd[k]);
        }
      }
    }
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      const int e = threadIdx.x + p * THREADS;
      const bool g = (gated >> p) & 1u;
      num[p] = (g || e >= E) ? R(0) : xi[(row0 + e / N) * N + (e % N)];
      den[p] = g ? R(0) : R(1);
    }
  }
  // after a redo den is 1 (kept) or 0 (guarded)
  recover_epilogue<R, PER, THREADS>(
      P, num, den, any ? R(0.5) : R(P.u_guard_f),
      [&](int p) {
        const int e = threadIdx.x + p * THREADS;
        return e < E ? (row0 + e / N) * N + (e % N) : -1LL;
      },
      xi, cout, ctr, red);
}

template <typename R, int N, bool INC>
cudaError_t rec_plane(const Problem& P, const Work<R>& w, R* xi, R* c, cudaStream_t s) {
  constexpr size_t smem = plane_rec_smem<R, N>();
  static SmemOptIn attr;
  cudaError_t e = opt_in_smem(attr, (const void*)k_ifft2_plane_recover<R, N, INC>, smem, true);
  if (e != cudaSuccess) return e;
  constexpr int C = plane_cluster<N>();
  e = launch_pdl_cluster(k_ifft2_plane_recover<R, N, INC>, dim3(C, (unsigned)P.m), dim3(THREADS), C, smem, s, P,
                         (const cx<R>*)w.prof, (const int*)w.slot, (const int*)w.cols, (const int*)w.ncol, w.u0, xi,
                         c, w.ctr, (const cx<R>*)w.tw);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

template <typename R, int N, int T>
cudaError_t rec_tiled(const Problem& P, const Work<R>& w, R* xi, R* c, cudaStream_t s, cudaEvent_t mid) {
  using GP = GatherPass<R, N, T>;
  using RP = RecPass<R, N, T>;
  // column chunks for the first GATHER_COLS active columns in the grid (the blocks loop
  // over more): the active columns are few in the usual case, and a grid of blocks that
  // return at once only delays the successor's launch (measured, 64-problem batch: 6.17
  // ms with every chunk in the grid, 6.07 with 32 columns; FP64 128^2 step +0.5 us)
  constexpr int NCH = (N + GP::GC - 1) / GP::GC, GZ = GATHER_COLS / GP::GC;
  const dim3 g1((P.m + GP::GL - 1) / GP::GL, 2 * P.n_omega, NCH < GZ ? NCH : GZ);
  cudaError_t e = launch_pdl(k_ifft_cols_gather<R, N, T>, g1, dim3(GP::NT), 0, s, P, (const cx<R>*)w.prof,
                             (const int*)w.slot, (const int*)w.cols, (const int*)w.ncol, w.t2, (const cx<R>*)w.tw);
  if (e != cudaSuccess) return e;
  if (mid) cudaEventRecord(mid, s);
  const long long nrows = (long long)P.m * N;
  const dim3 gr((unsigned)((nrows + RP::LINES - 1) / RP::LINES));
  e = w.u0 ? launch_pdl(k_ifft_rows_recover<R, N, true, T>, gr, dim3(RecForm<R, N, T>::NT), 0, s, P, (const cx<R>*)w.t2,
                        (const int*)w.colpos, (const int*)w.ncol, (const int*)w.colseg, w.u0, xi, c, w.ctr, (const cx<R>*)w.tw)
           : launch_pdl(k_ifft_rows_recover<R, N, false, T>, gr, dim3(RecForm<R, N, T>::NT), 0, s, P, (const cx<R>*)w.t2,
                        (const int*)w.colpos, (const int*)w.ncol, (const int*)w.colseg, w.u0, xi, c, w.ctr, (const cx<R>*)w.tw);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

template <typename R, int N>
cudaError_t rec_impl(const Problem& P, const Work<R>& w, R* xi, R* c, cudaStream_t s, cudaEvent_t mid) {
  // the mixed path: one pass unless asked otherwise (N = 96, 192 and 256 hold too many
  // values per thread for the cluster pass: two passes)
  if constexpr (sizeof(R) == 4 && N <= 128 && N != 96) {
    if (P.inverse_single) {
      if (mid) cudaEventRecord(mid, s);
      return w.u0 ? rec_plane<R, N, true>(P, w, xi, c, s) : rec_plane<R, N, false>(P, w, xi, c, s);
    }
  }
  return P.fft_tile == 1 ? rec_tiled<R, N, 1>(P, w, xi, c, s, mid) : rec_tiled<R, N, 0>(P, w, xi, c, s, mid);
}

}  // namespace

template <typename R>
cudaError_t launch_recover(const Problem& P, const Work<R>& w, R* xi, R* c, cudaStream_t s, cudaEvent_t mid) {
  switch (P.n) {
#define FL_CASE(K) case K: return rec_impl<R, K>(P, w, xi, c, s, mid);
    FL_SIZES(FL_CASE)
#undef FL_CASE
    default: return cudaErrorInvalidValue;
  }
}

template cudaError_t launch_recover<double>(const Problem&, const Work<double>&, double*, double*, cudaStream_t,
                                            cudaEvent_t);
template cudaError_t launch_recover<float>(const Problem&, const Work<float>&, float*, float*, cudaStream_t,
                                           cudaEvent_t);

}  // namespace fl
