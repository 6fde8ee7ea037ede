// Batched 1D FFTs of length N = 2^a 3^b on lines held in shared memory.
//
// The horizontal transform F_r of Sec. 2 (and its inverse, Algorithm 2 step 2)
// is a 2D DFT on the periodic N x N grid, done as two passes of 1D transforms:
// along x (contiguous rows) and along y (strided columns).  Two forms of a Stockham
// autosort FFT: fft_lines_io holds a line in registers at both ends (first stage from
// global memory, last stage to it) and crosses shared memory between stages only; fft_lines
// (the cluster kernels) works in place on a tile in shared memory: every stage reads all
// butterfly inputs into registers, synchronises, and writes the outputs back.
//
// Radices: 3 (once per factor 3), then the cap MAXR (16, 8 or 4) for as many powers of
// two as it covers, then one stage of 8, 4 or 2 for the rest: few stages, so few
// passes of the tile through shared memory.  The cap is set per kernel (measured):
// a large radix leaves threads idle when a tile has few butterflies.  For stage s with radix
// R and Ns = product of the earlier radices, butterfly j of a line reads elements
// j + r N/R, multiplies by w^(r (j mod Ns) N/(Ns R)) (w = exp(-2 pi i/N), conjugated
// for the inverse), applies the R-point DFT and writes element
// (j / Ns) Ns R + (j mod Ns) + r Ns.  Forward = unnormalised exp(-i...) DFT;
// inverse = unnormalised exp(+i...) DFT (the caller applies 1/N^2).
#pragma once

#include <type_traits>

#include "common.cuh"
#include "pair.cuh"

namespace fl {

__host__ __device__ constexpr int count_factor(int n, int f) { return (n % f == 0) ? 1 + count_factor(n / f, f) : 0; }
__host__ __device__ constexpr int strip(int n, int f) { return (n % f == 0) ? strip(n / f, f) : n; }

__host__ __device__ constexpr int log2i(int n) { return n > 1 ? 1 + log2i(n / 2) : 0; }

// MAXR (4, 8 or 16) caps the power-of-two radix
template <int N, int MAXR> struct FftPlan {
  static_assert(MAXR == 4 || MAXR == 8 || MAXR == 16, "radix cap 4, 8 or 16");
  static constexpr int n3 = count_factor(N, 3);
  static constexpr int p2 = count_factor(N, 2);
  static constexpr int q = log2i(MAXR);
  static constexpr int nbig = p2 / q;
  static constexpr int rest = 1 << (p2 % q);  // 1 (no further stage), 2, 4 or 8
  static constexpr int stages = n3 + nbig + (rest > 1 ? 1 : 0);
  static_assert(strip(strip(N, 2), 3) == 1, "N must be 2^a 3^b");
  __host__ __device__ static constexpr int radix(int s) { return s < n3 ? 3 : (s < n3 + nbig ? MAXR : rest); }
};

// cos and sin of 2 pi e / 16
__host__ __device__ constexpr double cos16(int e) {
  return (e & 15) == 0 ? 1.0 : (e & 15) == 1 ? 0.92387953251128674 : (e & 15) == 2 ? 0.70710678118654752
       : (e & 15) == 3 ? 0.38268343236508977 : (e & 15) == 4 ? 0.0 : (e & 15) == 5 ? -0.38268343236508977
       : (e & 15) == 6 ? -0.70710678118654752 : (e & 15) == 7 ? -0.92387953251128674 : (e & 15) == 8 ? -1.0
       : (e & 15) == 9 ? -0.92387953251128674 : (e & 15) == 10 ? -0.70710678118654752
       : (e & 15) == 11 ? -0.38268343236508977 : (e & 15) == 12 ? 0.0 : (e & 15) == 13 ? 0.38268343236508977
       : (e & 15) == 14 ? 0.70710678118654752 : 0.92387953251128674;
}
__host__ __device__ constexpr double sin16(int e) { return cos16(e + 12); }  // sin x = cos(x - pi/2)

// Line layouts inside a shared-memory tile.
//  ROW:  element i of line b at b*(N + N/S) + i + i/S    (rows of a plane), S = SKEW:
//        one padding element after every S keeps the stride-S writes of a radix-S
//        stage on distinct shared-memory banks (S = 0: b*N + i, no padding)
//  COL:  element i of line b sits at i*LINES + b         (columns of a plane tile)
enum class Lay { ROW, COL };

template <Lay L, int N, int LINES, int SKEW> struct LayIdx {
  static constexpr int STRIDE = (L == Lay::ROW && SKEW > 0) ? N + N / SKEW : N;
  static constexpr int ELEMS = LINES * STRIDE;  // elements of the tile, padding included
  __host__ __device__ __forceinline__ static int at(int b, int i) {
    return (L == Lay::ROW) ? b * STRIDE + i + (SKEW > 0 ? i / SKEW : 0) : i * LINES + b;
  }
  // thread-item -> (line, butterfly) so that neighbouring threads touch
  // neighbouring shared-memory words
  __device__ __forceinline__ static void map(int t, int nb, int& b, int& j) {
    if (L == Lay::ROW) { j = t % nb; b = t / nb; } else { b = t % LINES; j = t / LINES; }
  }
};

template <typename R, bool INV> struct Dft {
  using C = cx<R>;
  // a + rot90<I>(b)
  template <bool I> __device__ __forceinline__ static C add_rot(C a, C b) {
    return I ? mk<R>(a.x - b.y, a.y + b.x) : mk<R>(a.x + b.y, a.y - b.x);
  }
  __device__ __forceinline__ static void d2(C* v) {
    C a = v[0], b = v[1];
    v[0] = a + b; v[1] = a - b;
  }
  __device__ __forceinline__ static void d4(C* v) {
    C s02 = v[0] + v[2], d02 = v[0] - v[2];
    C s13 = v[1] + v[3], e = v[1] - v[3];
    v[0] = s02 + s13; v[2] = s02 - s13;
    v[1] = add_rot<INV>(d02, e); v[3] = add_rot<!INV>(d02, e);
  }
  // x w16^e, w16 = exp(-2 pi i/16) (conjugated for the inverse); e is a constant (w16^0
  // and w16^4 = -i cost no arithmetic: 10 of 170 FP64 operations of a 16-point DFT, on a
  // GPU where those bound the FP64 passes)
  __device__ __forceinline__ static C tw16(C x, int e) {
    if (e == 0) return x;
    if (e == 4) return rot90<INV>(x);
    if constexpr (std::is_same<R, f2>::value) {  // packed products are not contracted
      if (e == 8) return mk<R>(-x.x, -x.y);
      if (e == 12) return rot90<!INV>(x);
      const double cd = cos16(e), sd = INV ? sin16(e) : -sin16(e);
      return mk<R>(fma(x.y, R(-sd), x.x * R(cd)), fma(x.x, R(sd), x.y * R(cd)));
    }
    const R c = R(cos16(e)), sn = INV ? R(sin16(e)) : -R(sin16(e));
    return mk<R>(x.x * c - x.y * sn, x.x * sn + x.y * c);
  }
  // 8 points: 4-point DFTs of the even and odd inputs, X[k] = E[k] + w8^k O[k],
  // X[k + 4] = E[k] - w8^k O[k]
  __device__ __forceinline__ static void d8(C* v) {
    C e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    d4(e);
    d4(o);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const C t = tw16(o[k], 2 * k);
      v[k] = e[k] + t;
      v[k + 4] = e[k] - t;
    }
  }
  // 16 points as 4 x 4: with n = 4 n1 + n2 and k = k1 + 4 k2, 4-point DFTs over n1,
  // twiddles w16^(n2 k1), then 4-point DFTs over n2
  __device__ __forceinline__ static void d16(C* v) {
    C y[4][4];
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
      y[n2][0] = v[n2];
      y[n2][1] = v[n2 + 4];
      y[n2][2] = v[n2 + 8];
      y[n2][3] = v[n2 + 12];
      d4(y[n2]);
#pragma unroll
      for (int k1 = 1; k1 < 4; ++k1) y[n2][k1] = tw16(y[n2][k1], n2 * k1);
    }
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      C z[4] = {y[0][k1], y[1][k1], y[2][k1], y[3][k1]};
      d4(z);
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = z[k2];
    }
  }
  // 16 points of which only the first E and the last E (1 or 2) are not zero, as d16 would
  // transform them (the same operations on the same values, those with zeros left out: 44 or
  // 96 of 160)
  template <int E> __device__ __forceinline__ static void d16_edge(C* v) {
    const C a0 = v[0], b1 = v[15], a1 = E > 1 ? v[1] : v[0], b0 = E > 1 ? v[14] : v[15];
    C p0 = b0, p1 = b1;  // w4^(3 k1) b
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      constexpr bool PK = std::is_same<R, f2>::value;  // packed: w4^(3 k1) and the twiddle in one product
      const C t1 = tw16(a1, k1), t2 = tw16(PK ? b0 : p0, PK ? 14 * k1 % 16 : 2 * k1),
              t3 = tw16(PK ? b1 : p1, PK ? 15 * k1 % 16 : 3 * k1);
      if constexpr (E > 1) {
        C z[4] = {a0, t1, t2, t3};
        d4(z);
#pragma unroll
        for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = z[k2];
      } else {
        v[k1] = a0 + t3;
        v[k1 + 8] = a0 - t3;
        v[k1 + 4] = add_rot<!INV>(a0, t3);
        v[k1 + 12] = add_rot<INV>(a0, t3);
      }
      p0 = rot90<!INV>(p0);  // w4^3 = conj(w4)
      p1 = rot90<!INV>(p1);
    }
  }
  __device__ __forceinline__ static void d3(C* v) {
    // y1,2 = a0 - (a1+a2)/2 -/+ i (sqrt(3)/2)(a1 - a2)  (forward; signs swap for the inverse)
    const R h = R(0.86602540378443864676);
    if constexpr (sizeof(R) == 8) {  // 12 operations, the products fused into the sums
      const C s = v[1] + v[2], e = rot90<INV>(v[1] - v[2]);
      const C t = mk<R>(fma(R(-0.5), s.x, v[0].x), fma(R(-0.5), s.y, v[0].y));
      v[0] = v[0] + s;
      v[1] = mk<R>(fma(h, e.x, t.x), fma(h, e.y, t.y));
      v[2] = mk<R>(fma(R(-0.86602540378443864676), e.x, t.x), fma(R(-0.86602540378443864676), e.y, t.y));
    } else {
      C s = v[1] + v[2];
      C t = v[0] - R(0.5) * s;
      C d = h * rot90<INV>(v[1] - v[2]);
      v[0] = v[0] + s; v[1] = t + d; v[2] = t - d;
    }
  }
  // 12 points as 3 x 4 without twiddles (Good-Thomas): n = 4 n1 + 3 n2, k = 4 k1 + 9 k2
  // (mod 12) gives n k = 4 n1 k1 + 3 n2 k2 (mod 12)
  __device__ __forceinline__ static void d12(C* v) {
    C y[4][3];
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < 3; ++n1) y[n2][n1] = v[(4 * n1 + 3 * n2) % 12];
      d3(y[n2]);
    }
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) {
      C z[4] = {y[0][k1], y[1][k1], y[2][k1], y[3][k1]};
      d4(z);
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) v[(4 * k1 + 9 * k2) % 12] = z[k2];
    }
  }
  template <int RAD> __device__ __forceinline__ static void run(C* v) {
    if constexpr (RAD == 2) d2(v);
    else if constexpr (RAD == 3) d3(v);
    else if constexpr (RAD == 4) d4(v);
    else if constexpr (RAD == 8) d8(v);
    else if constexpr (RAD == 12) d12(v);
    else d16(v);
  }
};

template <typename R, int N, bool INV, int LINES, int THREADS, Lay L, int SKEW, int RAD, int NS>
__device__ __forceinline__ void fft_stage(cx<R>* buf, const cx<R>* tw) {
  using C = cx<R>;
  using IX = LayIdx<L, N, LINES, SKEW>;
  constexpr int NB = N / RAD;                 // butterflies per line
  constexpr int TOTAL = LINES * NB;
  constexpr int PER = (TOTAL + THREADS - 1) / THREADS;
  constexpr int STRIDE_TW = N / (NS * RAD);
  C v[PER][RAD];
  int out_b[PER], out_i[PER];
#pragma unroll
  for (int p = 0; p < PER; ++p) {
    const int t = threadIdx.x + p * THREADS;
    if (TOTAL % THREADS == 0 || t < TOTAL) {
      int b, j;
      IX::map(t, NB, b, j);
      const int k = j % NS;
#pragma unroll
      for (int r = 0; r < RAD; ++r) {
        C x = buf[IX::at(b, j + r * NB)];
        if (r > 0 && NS > 1) {
          C w = tw[r * k * STRIDE_TW];
          if (INV) w.y = -w.y;
          x = x * w;
        }
        v[p][r] = x;
      }
      if constexpr (RAD == 2) Dft<R, INV>::d2(v[p]);
      else if constexpr (RAD == 4) Dft<R, INV>::d4(v[p]);
      else if constexpr (RAD == 8) Dft<R, INV>::d8(v[p]);
      else if constexpr (RAD == 16) Dft<R, INV>::d16(v[p]);
      else Dft<R, INV>::d3(v[p]);
      out_b[p] = b;
      out_i[p] = (j / NS) * NS * RAD + k;
    }
  }
  __syncthreads();
#pragma unroll
  for (int p = 0; p < PER; ++p) {
    const int t = threadIdx.x + p * THREADS;
    if (TOTAL % THREADS == 0 || t < TOTAL) {
#pragma unroll
      for (int r = 0; r < RAD; ++r) buf[IX::at(out_b[p], out_i[p] + r * NS)] = v[p][r];
    }
  }
  __syncthreads();
}

// stage S of the plan, with NS = product of the earlier radices (compile-time)
template <typename R, int N, bool INV, int LINES, int THREADS, Lay L, int SKEW, int MAXR, int S, int NS>
struct FftStages {
  __device__ __forceinline__ static void run(cx<R>* buf, const cx<R>* tw) {
    if constexpr (S < FftPlan<N, MAXR>::stages) {
      constexpr int RAD = FftPlan<N, MAXR>::radix(S);
      fft_stage<R, N, INV, LINES, THREADS, L, SKEW, RAD, NS>(buf, tw);
      FftStages<R, N, INV, LINES, THREADS, L, SKEW, MAXR, S + 1, NS * RAD>::run(buf, tw);
    }
  }
};

// Transform all LINES lines of the tile in place.  `tw` holds w^j, j < N
// (w = exp(-2 pi i/N)), in shared or global memory.  Must be called by all
// THREADS threads of the block; contains __syncthreads().
template <typename R, int N, bool INV, int LINES, int THREADS, Lay L, int MAXR, int SKEW = 0>
__device__ __forceinline__ void fft_lines(cx<R>* buf, const cx<R>* tw) {
  FftStages<R, N, INV, LINES, THREADS, L, SKEW, MAXR, 0, 1>::run(buf, tw);
}

// ---- transforms between global memory and registers ---------------------------
// The passes below hold a line in registers at both ends: the first stage's inputs are
// loaded straight from global memory in butterfly order (element j + r N/RAD, neighbouring
// threads on neighbouring elements), the last stage's outputs (element k + r N/RAD) leave
// from registers.  A two-stage length crosses shared memory once and meets one barrier;
// staging the tile in shared memory first and last took three crossings and four barriers.

// Plans of these passes.  3-smooth lengths end in a 12-point stage (no inner twiddles):
// 192 = 16 x 12, one crossing, where 3 x 16 x 4 takes two and 20% more operations.
// DENSE32 keeps FftPlan's factors: the FP32 transforms of the derivatives, whose FP64
// sums (Phi) follow the rounding of the transform.
template <int N, int MAXR, bool DENSE32> struct IoPlan {
  static constexpr bool R12 = !DENSE32 && N % 12 == 0 && N / 12 <= MAXR && (N / 12 & (N / 12 - 1)) == 0;
  static constexpr int stages = R12 ? (N > 12 ? 2 : 1) : FftPlan<N, MAXR>::stages;
  __host__ __device__ static constexpr int radix(int s) {
    return R12 ? (s == stages - 1 ? 12 : N / 12) : FftPlan<N, MAXR>::radix(s);
  }
  // product of the radices before stage s
  __host__ __device__ static constexpr int ns(int s) { return s == 0 ? 1 : ns(s - 1) * radix(s - 1); }
  // twiddles by stage: entry r NS + k of stage s >= 1 at off(s), w^(r k N/(NS RAD)) -- a row of
  // consecutive k per r, so that neighbouring butterflies read neighbouring entries
  __host__ __device__ static constexpr int off(int s) { return s <= 1 ? 0 : off(s - 1) + ns(s - 1) * radix(s - 1); }
  static constexpr int tw_elems = stages > 1 ? off(stages - 1) + ns(stages - 1) * radix(stages - 1) : 1;
};

template <typename R, class PL, int N, int THREADS, int S = 1>
__device__ __forceinline__ void load_stage_twiddles(cx<R>* tws, const cx<R>* __restrict__ tw) {
  if constexpr (S < PL::stages) {
    constexpr int NS = PL::ns(S), RAD = PL::radix(S), ST = N / (NS * RAD);
    for (int e = threadIdx.x; e < NS * RAD; e += THREADS) tws[PL::off(S) + e] = tw[(e / NS) * (e % NS) * ST];
    load_stage_twiddles<R, PL, N, THREADS, S + 1>(tws, tw);
  }
}

// the same table, each entry for both values of a pair
template <class PL, int N, int THREADS, int S = 1>
__device__ __forceinline__ void load_stage_twiddles_pairs(cf2* tws, const float2* __restrict__ tw) {
  if constexpr (S < PL::stages) {
    constexpr int NS = PL::ns(S), RAD = PL::radix(S), ST = N / (NS * RAD);
    for (int e = threadIdx.x; e < NS * RAD; e += THREADS) {
      const float2 w = tw[(e / NS) * (e % NS) * ST];
      tws[PL::off(S) + e] = pair_of(w, w);
    }
    load_stage_twiddles_pairs<PL, N, THREADS, S + 1>(tws, tw);
  }
}

// the RAD inputs of butterfly j of line b at stage S >= 1 from the tile, twiddled and transformed
template <typename R, class PL, int N, bool INV, int LINES, Lay L, int SKEW, int S>
__device__ __forceinline__ void io_butterfly(const cx<R>* buf, const cx<R>* tws, int b, int j, cx<R>* v) {
  using IX = LayIdx<L, N, LINES, SKEW>;
  constexpr int RAD = PL::radix(S), NS = PL::ns(S), NB = N / RAD;
  const int k = j % NS;
#pragma unroll
  for (int r = 0; r < RAD; ++r) {
    cx<R> x = buf[IX::at(b, j + r * NB)];
    if (r > 0) {
      cx<R> w = tws[PL::off(S) + r * NS + k];
      if constexpr (std::is_same<R, f2>::value) {
        x = INV ? mk<R>(fma(x.y, w.y, x.x * w.x), x.y * w.x - x.x * w.y) : x * w;
      } else {
        if (INV) w.y = -w.y;
        x = x * w;
      }
    }
    v[r] = x;
  }
  Dft<R, INV>::template run<RAD>(v);
}

// stages S .. stages - 2 in place in the tile
template <typename R, class PL, int N, bool INV, int LINES, int THREADS, Lay L, int SKEW, int S>
__device__ __forceinline__ void io_middle(cx<R>* buf, const cx<R>* tws) {
  if constexpr (S < PL::stages - 1) {
    using IX = LayIdx<L, N, LINES, SKEW>;
    constexpr int RAD = PL::radix(S), NS = PL::ns(S), NB = N / RAD, TOTAL = LINES * NB;
    constexpr int PER = (TOTAL + THREADS - 1) / THREADS;
    cx<R> v[PER][RAD];
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      const int t = threadIdx.x + p * THREADS;
      if (TOTAL % THREADS == 0 || t < TOTAL) {
        int b, j;
        IX::map(t, NB, b, j);
        io_butterfly<R, PL, N, INV, LINES, L, SKEW, S>(buf, tws, b, j, v[p]);
      }
    }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      const int t = threadIdx.x + p * THREADS;
      if (TOTAL % THREADS == 0 || t < TOTAL) {
        int b, j;
        IX::map(t, NB, b, j);
        const int o = (j / NS) * NS * RAD + j % NS;
#pragma unroll
        for (int r = 0; r < RAD; ++r) buf[IX::at(b, o + r * NS)] = v[p][r];
      }
    }
    __syncthreads();
    io_middle<R, PL, N, INV, LINES, THREADS, L, SKEW, S + 1>(buf, tws);
  }
}

// First stage: ld(b, i) gives element i of line b; its outputs go to the tile (then a
// barrier and the middle stages), ready for the last stage.  Only for plans of two stages
// or more.  PRE: an index load first: the thread's ld.pre(b, i) (ints), then its ld(b, i, index).
// TILE: ld reads the same tile (a barrier between the loads and the results).
template <typename R, class PL, int N, bool INV, int LINES, int THREADS, Lay L, int SKEW, bool PRE = false,
          bool TILE = false, class Ld>
__device__ __forceinline__ void io_first(cx<R>* buf, const cx<R>* tws, Ld ld) {
  using IX = LayIdx<L, N, LINES, SKEW>;
  constexpr int RAD = PL::radix(0), NB = N / RAD, TOTAL = LINES * NB;
  constexpr int PER = (TOTAL + THREADS - 1) / THREADS;
  cx<R> v[PER][RAD];
  {  // every load of the thread first
    int at[PRE ? PER : 1][PRE ? RAD : 1];
    if constexpr (PRE) {
#pragma unroll
      for (int p = 0; p < PER; ++p) {
        const int t = threadIdx.x + p * THREADS;
        if (TOTAL % THREADS == 0 || t < TOTAL) {
          int b, j;
          IX::map(t, NB, b, j);
#pragma unroll
          for (int r = 0; r < RAD; ++r) at[p][r] = ld.pre(b, j + r * NB);
        }
      }
    }
#pragma unroll
    for (int p = 0; p < PER; ++p) {
      const int t = threadIdx.x + p * THREADS;
      if (TOTAL % THREADS == 0 || t < TOTAL) {
        int b, j;
        IX::map(t, NB, b, j);
#pragma unroll
        for (int r = 0; r < RAD; ++r) {
          if constexpr (PRE) v[p][r] = ld(b, j + r * NB, at[p][r]);
          else v[p][r] = ld(b, j + r * NB);
        }
      }
    }
  }
  if constexpr (TILE) __syncthreads();
#pragma unroll
  for (int p = 0; p < PER; ++p) {
    const int t = threadIdx.x + p * THREADS;
    if (TOTAL % THREADS == 0 || t < TOTAL) {
      int b, j;
      IX::map(t, NB, b, j);
      Dft<R, INV>::template run<RAD>(v[p]);
#pragma unroll
      for (int r = 0; r < RAD; ++r) buf[IX::at(b, j * RAD + r)] = v[p][r];
    }
  }
  __syncthreads();
  io_middle<R, PL, N, INV, LINES, THREADS, L, SKEW, 1>(buf, tws);
}

// The last stage: st(b, i, value) takes the results (its own inputs' places in the tile are free).
template <typename R, class PL, int N, bool INV, int LINES, int THREADS, Lay L, int SKEW, class St>
__device__ __forceinline__ void io_last(const cx<R>* buf, const cx<R>* tws, St st) {
  using IX = LayIdx<L, N, LINES, SKEW>;
  constexpr int S = PL::stages - 1, RAD = PL::radix(S), NB = N / RAD, TOTAL = LINES * NB;
  for (int t = threadIdx.x; t < TOTAL; t += THREADS) {
    int b, j;
    IX::map(t, NB, b, j);
    cx<R> v[RAD];
    io_butterfly<R, PL, N, INV, LINES, L, SKEW, S>(buf, tws, b, j, v);
#pragma unroll
    for (int r = 0; r < RAD; ++r) st(b, j + r * NB, v[r]);
  }
}

// Transform LINES lines: ld(b, i) -> element i of line b, st(b, i, value) takes the results.
// Called by all THREADS threads; the twiddles tws (load_stage_twiddles) need no barrier
// before it when the plan has a barrier (two stages or more).  Safe in place: every load is
// made before the barrier, every store after it (one stage: a thread owns whole lines).
template <typename R, class PL, int N, bool INV, int LINES, int THREADS, Lay L, int SKEW, bool PRE = false, class Ld,
          class St>
__device__ __forceinline__ void fft_lines_io(cx<R>* buf, const cx<R>* tws, Ld ld, St st) {
  using IX = LayIdx<L, N, LINES, SKEW>;
  constexpr int S = PL::stages - 1, RAD = PL::radix(S), NB = N / RAD, TOTAL = LINES * NB;
  if constexpr (S == 0) {
    for (int b = threadIdx.x; b < LINES; b += THREADS) {
      cx<R> v[RAD];
#pragma unroll
      for (int r = 0; r < RAD; ++r) {
        if constexpr (PRE) v[r] = ld(b, r, ld.pre(b, r));
        else v[r] = ld(b, r);
      }
      Dft<R, INV>::template run<RAD>(v);
#pragma unroll
      for (int r = 0; r < RAD; ++r) st(b, r, v[r]);
    }
  } else {
    io_first<R, PL, N, INV, LINES, THREADS, L, SKEW, PRE>(buf, tws, ld);
    io_last<R, PL, N, INV, LINES, THREADS, L, SKEW>(buf, tws, st);
  }
}

}  // namespace fl
