// Forward data generator on the device.
//
// Single scattering (Born): Algorithm 1 (Sec. 3) stopped before its first
// iteration, so U~ = U~0 and eq. (7) gives
//   V~ = F_r[xi F^-1 U~0] = F_r[xi u0],   W~_k = omega^2 sum_l h_z K_nu(z_k - z'_l) V~_l,
//   W = F^-1[W~]  on the data planes.
// Full scattering: Algorithm 1 itself, the fixed point of eq. (6),
//   U~_{n+1} = U~0 + omega^2 T_nu F_r[xi F^-1 U~_n],  T_nu[l, l'] = h_z K_nu(z'_l - z'_l'),
// stopped when ||U~_{n+1} - U~_n|| <= rtol ||U~0|| (Sec. 5.1), then eq. (7) with the
// converged field.  T_nu is applied as in eq. (9) of the inverse: with q = e^{i k_z h_z},
// h_z K_nu(z'_l - z'_l') = gamma q^|l - l'| / omega^2, a forward and a backward first-order
// recurrence over the planes, one thread per mode.
// The incident field is the plane wave u0 = exp(-i k0 z).  As in the solve, every
// data plane lies above X, so exp(i k_z (z_k - z'_l)) = exp(i k_z (z_k - z'_top)) *
// exp(i k_z (z'_top - z'_l)) and the sum over l is shared by all k.  Grazing modes
// (|nu| = k0) carry K = 0.
#include <math.h>

#include <complex>
#include <vector>

#include <string.h>

#include "modes.cuh"
#include "pipeline.cuh"

namespace fl {

namespace {

// V = xi u0 on X (omega^2 sits in the kernel factor), u0 the given incident field
// [n_omega][M][N][N]
template <typename R>
__global__ void k_source(Problem P, const R* __restrict__ xi, const cx<R>* __restrict__ u0i, cx<R>* __restrict__ src) {
  const long long per = (long long)P.m * P.n * P.n;
  const long long total = per * P.n_omega;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const R x = xi[e % per];
    const cx<R> u = u0i[e];
    src[e] = mk<R>(x * u.x, x * u.y);
  }
}

// U~0 of point sources on the X planes (periodic model, Sec. 5): thread per (omega, l, nu),
// U~0 = (N^2/L^2) sum_s a_s K_nu(z'_l - z_s) e^{-i nu.(r_s - x0)}, K_nu(dz) = -i e^{i k_z|dz|}/(2 k_z),
// x0 = -L/2 (the grid's first node); zero on grazing modes
template <typename R>
__global__ void k_point_sources(Problem P, const double* __restrict__ spec, int n_src, cx<R>* __restrict__ ut) {
  const int N = P.n;
  const long long N2 = (long long)N * N;
  const long long total = (long long)P.n_omega * P.m * N2;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const long long pl = e / N2;
    const int nu = (int)(e - pl * N2);
    const int om = (int)(pl / P.m), l = (int)(pl - (long long)om * P.m);
    const int i2 = nu / N, i1 = nu - i2 * N;
    const int m1 = i1 < N / 2 ? i1 : i1 - N, m2 = i2 < N / 2 ? i2 : i2 - N;
    const int msq = m1 * m1 + m2 * m2;
    double2 acc = make_double2(0.0, 0.0);
    if (!(msq >= P.graz_lo[om] && msq <= P.graz_hi[om])) {
      const double k0 = P.k0[om];
      const double q = k0 * k0 - P.kn * P.kn * (double)msq;
      const double2 kz = q >= 0.0 ? make_double2(sqrt(q), 0.0) : make_double2(0.0, sqrt(-q));
      // -i / (2 k_z): k_z real -> (0, -1/(2 k_z)); k_z = i kappa -> (-1/(2 kappa), 0)
      const double2 g = q >= 0.0 ? make_double2(0.0, -0.5 / kz.x) : make_double2(-0.5 / kz.y, 0.0);
      const double zl = P.z1 + (l + 0.5) * P.hz, x0 = -0.5 * P.period;
      const double nu1 = P.kn * m1, nu2 = P.kn * m2;
      for (int j = 0; j < n_src; ++j) {
        const double* sp = spec + 4 * j;
        const double2 ez = exp_ikz_inline(kz, sp[2] - zl);  // sources above X: |dz| = z_s - z'_l
        double sn, cs;
        sincos(-(nu1 * (sp[0] - x0) + nu2 * (sp[1] - x0)), &sn, &cs);
        acc = acc + sp[3] * (ez * make_double2(cs, sn));
      }
      acc = (double)N2 / (P.period * P.period) * (g * acc);
    }
    ut[e] = from_d<R>(acc);
  }
}

// ---- eq. (7): W~_k = E_k sum_l P_l V~_l on every mode ---------------------------
// P_l = q^(M-1-l): the planes are taken in blocks of HB from the lowest (the first may be
// short), a Horner recurrence in q inside a block, the block's top P by its own exponential.
// The data planes likewise, in blocks of HB, when they are uniform to rounding: E_k from the
// block's first plane by powers of e^{i k_z dz}, times 1 + i k_z d_k for the offset d_k of the
// given height from the uniform one (|k_z d_k| < 1e-9, so its square is below rounding).
// Otherwise one exponential per plane.  So no power is further than HB - 1 products from an
// exponential, whose own rounding is of that size.
//
// FP64 arithmetic bounds this kernel (an FP64 exp is ~40 instructions, a sincos ~60, at 1/64
// of the FP32 rate), so nothing is evaluated twice: the modes (+-m1, +-m2) share k_z, hence
// q and every E_k.  A block takes 32 quadrant modes (m1, m2 >= 0), one warp per sign pair; the
// four warps deal the exponentials among themselves through shared memory, then each sums its
// own modes.  An evanescent mode (q, E real) takes real products.  Before, one thread per
// mode took an exp and a sincos per plane: 192^2, 37 + 19 planes, 5 frequencies (FP64, REAL)
// 1067 us -> 194 us (85% of the FP64 rate), 128^2, 64 + 32 planes 363 us -> 44 us.
//
// REAL (the plane incident wave): V~_l = e^{-i k0 z'_l} F[xi_l], and the transform of the real planes
// xi_l, half of its columns (launch_fft2_real), serves every frequency (FG of them per block, so that it
// is read once for them).  The phase joins q: rho = q e^{i k0 h_z}.  Otherwise vt holds V~ per
// frequency.
constexpr int HB = 8;   // planes per block
constexpr int FG = 2;   // frequencies per thread block (REAL; 4 left the SMs unevenly loaded)
constexpr int EK = 32;  // data planes per pass over the exponentials (planes not uniform)

struct DataPlanes {  // uniform spacing (0: not uniform) and the offsets from it
  double dz;
  double off[MAX_M1];
};

__device__ __forceinline__ double2 kz_vec(bool prop, double kz) {
  return prop ? make_double2(kz, 0.0) : make_double2(0.0, kz);
}

// a E_k for the planes of out, E_k on lanes in shared memory: block heads and the step (uniform
// planes, UNI) or one per plane.  CPLX: the warp holds a propagating mode.
template <typename R, bool UNI, bool CPLX>
__device__ __forceinline__ void put_data(const Problem& P, const DataPlanes& D, const double2 (*ex)[32], int lane,
                                         int k0, int kn, double2 kz, double2 a, cx<R>* out, long long N2) {
  if constexpr (UNI) {
    const double2 step = ex[0][lane];
    double2 e = make_double2(0.0, 0.0);
    for (int k = 0; k < P.m1; ++k) {
      const double d = D.off[k];
      if (k % HB == 0) e = ex[1 + k / HB][lane];
      else e = CPLX ? e * step : make_double2(e.x * step.x, 0.0);
      if constexpr (CPLX) {  // 1 + i k_z d
        const double2 f = make_double2(fma(-kz.y, d, 1.0), kz.x * d);
        out[k * N2] = from_d<R>((e * f) * a);
      } else {
        const double c = fma(-kz.y * d, e.x, e.x);
        out[k * N2] = from_d<R>(make_double2(c * a.x, c * a.y));
      }
    }
  } else {
    for (int j = 0; j < kn; ++j) {
      const double2 x = ex[j][lane];
      out[(k0 + j) * N2] = from_d<R>(CPLX ? x * a : make_double2(x.x * a.x, x.x * a.y));
    }
  }
}

template <bool REAL> constexpr int apply_nf() { return REAL ? FG : 1; }
__host__ __device__ inline int apply_blocks(int m) { return (m + HB - 1) / HB; }
// shared memory: heads [NF][nbk], q [NF], phases [NF][nbk] and the data exponentials
template <bool REAL> size_t apply_smem(int m) {
  return sizeof(double2) * ((size_t)apply_nf<REAL>() * ((apply_blocks(m) + 1) * 32 + apply_blocks(m)) + EK * 32);
}

template <typename R, bool REAL, bool UNI>
__global__ void __launch_bounds__(128)
k_apply_data(Problem P, DataPlanes D, const cx<R>* __restrict__ vt, cx<R>* __restrict__ wt) {
  constexpr int NF = apply_nf<REAL>();
  extern __shared__ __align__(16) unsigned char apply_raw[];
  const int N = P.n, M = P.m, H = N / 2 + 1;
  const int nbk = apply_blocks(M);  // block b ends at plane M - 1 - HB (nbk - 1 - b)
  double2 (*ex)[32] = reinterpret_cast<double2 (*)[32]>(apply_raw);
  double2 (*hd)[32] = ex + EK;              // [NF][nbk]
  double2 (*rs)[32] = hd + NF * nbk;        // [NF]
  double2* phs = &rs[NF][0];                // [NF][nbk]
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long N2 = (long long)N * N;
  const int e = blockIdx.x * 32 + lane;
  const bool in = e < H * H;
  const int m2 = in ? e / H : 0, m1 = in ? e - m2 * H : 0;
  // this warp's mode (+-m1, +-m2); index N/2 is its own mirror image, as is 0
  const bool neg1 = w & 1, neg2 = w & 2;
  const bool valid = in && !(neg1 && (m1 == 0 || m1 == N / 2)) && !(neg2 && (m2 == 0 || m2 == N / 2));
  const int i1 = neg1 ? (N - m1) % N : m1, i2 = neg2 ? (N - m2) % N : m2;
  const long long nu = (long long)i2 * N + i1;
  const int msq = m1 * m1 + m2 * m2;
  const double ztop = P.z1 + (M - 0.5) * P.hz;
  const int om0 = REAL ? blockIdx.y * FG : blockIdx.y;
  const int nf = REAL ? min(FG, P.n_omega - om0) : 1;
  if (REAL) {  // e^{-i k0 z'} of the block tops and e^{i k0 h_z}
    for (int t = threadIdx.x; t < nf * (nbk + 1); t += 128) {
      const int f = t / (nbk + 1), b = t - f * (nbk + 1);
      double s, c;
      sincos(b < nbk ? -P.k0[om0 + f] * (P.z1 + (M - 1 - HB * (nbk - 1 - b) + 0.5) * P.hz) : P.k0[om0 + f] * P.hz, &s,
             &c);
      if (b < nbk) phs[f * nbk + b] = make_double2(c, s);
      else ex[f][0] = make_double2(c, s);
    }
    __syncthreads();
  }
  double kz[NF], gam[NF];  // |k_z| and |gamma| with its sign (gamma = i gam or gam)
  unsigned propm = 0;
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    if (f >= nf) break;
    const int om = om0 + f;
    const bool grazing = msq >= P.graz_lo[om] && msq <= P.graz_hi[om];  // k_z = 0: excluded, a placeholder
    const double qq = P.k0[om] * P.k0[om] - P.kn * P.kn * (double)msq;
    const double r = grazing ? 1.0 : rsqrt64(fabs(qq));
    kz[f] = grazing ? 1.0 : sqrt_from_rsqrt(fabs(qq), r);
    gam[f] = grazing ? 0.0 : (REAL ? -0.5 : -1.0) * P.g0[om] * r;  // REAL: vt is twice the transform
    propm |= (qq >= 0.0 ? 1u : 0u) << f;
  }
  {
    int it = 0;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      if (f >= nf) break;
      const double2 k = kz_vec(propm >> f & 1u, kz[f]);
      for (int b = 0; b <= nbk; ++b, ++it) {
        if ((it & 3) != w) continue;
        double2 x = exp_ikz_inline(k, b < nbk ? HB * (nbk - 1 - b) * P.hz : P.hz);
        if (REAL) x = x * (b < nbk ? phs[f * nbk + b] : ex[f][0]);
        if (b < nbk) hd[f * nbk + b][lane] = x;
        else rs[f][lane] = x;
      }
    }
  }
  __syncthreads();
  double2 acc[NF];
#pragma unroll
  for (int f = 0; f < NF; ++f) acc[f] = make_double2(0.0, 0.0);
  if constexpr (REAL) {
    double2 rho[NF], blk[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) {
      rho[f] = f < nf ? rs[f][lane] : make_double2(0.0, 0.0);
      blk[f] = make_double2(0.0, 0.0);
    }
    if (valid) {
      // a mode with m1 < 0 from its mirror image, which is its conjugate
      const int HS = real_stride(N);
      const long long NH = (long long)N * HS;
      const cx<R>* src = vt + (long long)(neg1 ? (N - i2) % N : i2) * HS + m1;
      for (int b = 0, l0 = M - HB * nbk; b < nbk; ++b, l0 += HB) {  // (the first block may be short)
        cx<R> v[HB];
#pragma unroll
        for (int j = 0; j < HB; ++j) v[j] = l0 + j >= 0 ? src[(l0 + j) * NH] : czero<R>();
#pragma unroll
        for (int j = 0; j < HB; ++j) {
          if (l0 + j < 0) continue;
          double2 x = to_d(v[j]);
          if (neg1) x.y = -x.y;
#pragma unroll
          for (int f = 0; f < NF; ++f)
            if (f < nf) blk[f] = rho[f] * blk[f] + x;
        }
#pragma unroll
        for (int f = 0; f < NF; ++f) {
          if (f < nf) acc[f] = acc[f] + hd[f * nbk + b][lane] * blk[f];
          blk[f] = make_double2(0.0, 0.0);
        }
      }
    }
  } else {
    const double2 q = rs[0][lane];
    const bool cplx = __any_sync(0xffffffffu, propm);
    if (valid) {
      const cx<R>* src = vt + (long long)om0 * M * N2 + nu;
      for (int b = 0, l = 0; b < nbk; ++b) {
        const int l1 = M - HB * (nbk - 1 - b);
        double2 blk = make_double2(0.0, 0.0);
        if (cplx) {
#pragma unroll 4
          for (; l < l1; ++l) blk = q * blk + to_d(src[l * N2]);
          acc[0] = acc[0] + hd[b][lane] * blk;
        } else {
#pragma unroll 4
          for (; l < l1; ++l) {
            const double2 v = to_d(src[l * N2]);
            blk = make_double2(fma(q.x, blk.x, v.x), fma(q.x, blk.y, v.y));
          }
          const double h = hd[b][lane].x;
          acc[0] = make_double2(fma(h, blk.x, acc[0].x), fma(h, blk.y, acc[0].y));
        }
      }
    }
  }
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    if (f >= nf) break;
    const int om = om0 + f;
    const bool prop = propm >> f & 1u;
    const bool cplx = __any_sync(0xffffffffu, prop);
    const double2 k = kz_vec(prop, kz[f]);
    const double g = gam[f];
    const double2 a = prop ? make_double2(-g * acc[f].y, g * acc[f].x) : make_double2(g * acc[f].x, g * acc[f].y);
    cx<R>* out = wt + (long long)om * P.m1 * N2 + nu;
    for (int k0 = 0; k0 < P.m1; k0 += UNI ? MAX_M1 : EK) {
      const int kn = UNI ? P.m1 : min(EK, P.m1 - k0);
      const int items = UNI ? 1 + (P.m1 + HB - 1) / HB : kn;  // UNI: the step, then the block heads
      __syncthreads();
      for (int j = w; j < items; j += 4)
        ex[j][lane] = exp_ikz_inline(k, UNI ? (j == 0 ? D.dz : P.zy[HB * (j - 1)] - ztop) : P.zy[k0 + j] - ztop);
      __syncthreads();
      if (valid) {
        if (cplx) put_data<R, UNI, true>(P, D, ex, lane, k0, kn, k, a, out, N2);
        else put_data<R, UNI, false>(P, D, ex, lane, k0, kn, k, a, out, N2);
      }
    }
  }
}

// the offsets of the data planes from uniform heights in blocks of HB (off[k] is taken from
// the block's first plane); false when they are not uniform to rounding
inline bool uniform_planes(const Problem& P, DataPlanes* D) {
  const int m1 = P.m1;
  D->dz = m1 > 1 ? (P.zy[m1 - 1] - P.zy[0]) / (m1 - 1) : 0.0;
  if (m1 < HB || !(D->dz > 0.0)) return false;  // few planes: their own exponentials
  double kmax = P.kn * P.n;  // above every |k_z| of the grid and the frequencies
  for (int j = 0; j < P.n_omega; ++j) kmax = fmax(kmax, P.k0[j]);
  for (int k = 0; k < m1; ++k) {
    const int h = k - k % HB;
    D->off[k] = (double)((long double)P.zy[k] - P.zy[h] - (long double)(k - h) * D->dz);
    if (!(fabs(D->off[k]) * kmax < 1e-9)) return false;
  }
  return true;
}

template <typename R, bool REAL, bool UNI>
cudaError_t apply_variant(const Problem& P, const DataPlanes& D, const cx<R>* vt, cx<R>* wt, cudaStream_t s) {
  const size_t smem = apply_smem<REAL>(P.m);
  static SmemOptIn attr;
  const cudaError_t e = opt_in_smem(attr, (const void*)k_apply_data<R, REAL, UNI>, apply_smem<REAL>(MAX_M));
  if (e != cudaSuccess) return e;
  const int H = P.n / 2 + 1;
  const dim3 g((unsigned)((H * H + 31) / 32), (P.n_omega + apply_nf<REAL>() - 1) / apply_nf<REAL>());
  k_apply_data<R, REAL, UNI><<<g, 128, smem, s>>>(P, D, vt, wt);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_apply_data(const Problem& P, const cx<R>* vt, bool real, cx<R>* wt, cudaStream_t s) {
  DataPlanes D;
  memset(&D, 0, sizeof(D));
  if (uniform_planes(P, &D))
    return real ? apply_variant<R, true, true>(P, D, vt, wt, s) : apply_variant<R, false, true>(P, D, vt, wt, s);
  return real ? apply_variant<R, true, false>(P, D, vt, wt, s) : apply_variant<R, false, false>(P, D, vt, wt, s);
}

}  // namespace

template <typename R>
cudaError_t launch_point_sources(const Problem& P, const double* spec, int n_src, cx<R>* u0, const cx<R>* tw,
                                 cudaStream_t s) {
  k_point_sources<R><<<2048, 256, 0, s>>>(P, spec, n_src, u0);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_fft2_dense<R>(u0, u0, P.n, (long long)P.n_omega * P.m, true, tw, s);
}

template cudaError_t launch_point_sources<double>(const Problem&, const double*, int, double2*, const double2*,
                                                  cudaStream_t);
template cudaError_t launch_point_sources<float>(const Problem&, const double*, int, float2*, const float2*,
                                                 cudaStream_t);

template <typename R>
cudaError_t launch_forward_born(const Problem& P, const R* xi, const cx<R>* u0, cx<R>* src, cx<R>* W,
                                const cx<R>* tw, cudaStream_t s) {
  cudaError_t e;
  if (u0) {
    k_source<R><<<1024, 256, 0, s>>>(P, xi, u0, src);
    e = launch_fft2_dense<R>(src, src, P.n, (long long)P.n_omega * P.m, false, tw, s);
  } else {
    // the plane wave is constant on a plane: one transform of the real planes xi_l instead of one of
    // xi_l e^{-i k0 z'_l} per plane and frequency
    e = launch_fft2_real<R>(xi, src, P.n, P.m, tw, s);
  }
  if (e != cudaSuccess) return e;
  if ((e = launch_apply_data<R>(P, src, u0 == nullptr, W, s)) != cudaSuccess) return e;
  return launch_fft2_dense<R>(W, W, P.n, (long long)P.n_omega * P.m1, true, tw, s);
}

template cudaError_t launch_forward_born<double>(const Problem&, const double*, const double2*, double2*, double2*,
                                                 const double2*, cudaStream_t);
template cudaError_t launch_forward_born<float>(const Problem&, const float*, const float2*, float2*, float2*,
                                                const float2*, cudaStream_t);


// ---- Algorithm 1 (fixed point of eq. 6) -------------------------------------
namespace {

constexpr int FP_T = 256;  // threads per block of the fixed-point kernels

// U~0 of one frequency: N^2 exp(-i k0 z'_l) at nu = 0 (the rest is zeroed by the caller), also
// kept in inc [M] for k_interior (M sincos on the lanes of one block would outlast the rest of
// its grid)
template <typename R>
__global__ void k_incident(Problem P, cx<R>* __restrict__ ut, cx<R>* __restrict__ inc) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l < P.m) {
    double s, c;
    sincos(-P.k0[0] * (P.z1 + (l + 0.5) * P.hz), &s, &c);
    const double n2 = (double)P.n * P.n;
    inc[l] = from_d<R>(make_double2(n2 * c, n2 * s));
    ut[(long long)l * P.n * P.n] = inc[l];
  }
}

// *out = sum of n partials (one block, a fixed order); out may be mapped host memory
__global__ void __launch_bounds__(256) k_sum_partials(const double* __restrict__ partial, int n, double* out) {
  __shared__ double red[8];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) s += partial[i];
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) s += red[w];
    *out = s;
  }
}

// omega^2 T_nu V~ for every mode of one frequency: gamma (F + B) with
// F_l = q F_{l-1} + V~_l, B_l = q H_{l+1}, H_l = V~_l + q H_{l+1}.
// STEP (a step of Algorithm 1): ut <- U~0 + gamma (F + B) and the block partial of
// ||U~_{n+1} - U~_n||^2 in a fixed order; otherwise ut <- gamma (F + B).
// u0t (STEP only, may be null): U~0 of a given incident field on every mode; null for the
// plane wave, whose U~0 is N^2 exp(-i k0 z'_l) at nu = 0 alone.
//
// A block holds 32 modes (lanes) and cuts the planes into IG chunks of CP, one per warp: each
// warp runs its chunk's two recurrences from zero, the chunks' end values meet in shared memory,
// and each warp replays its chunk from the values that enter it.  One thread per mode ran all
// 2 M dependent steps at one FP64 instruction per 64 cycles, in N^2/256 blocks (64 SMs at N =
// 128); the chunks cost 4 of 16 FP64 instructions per plane and fill the chip.  An evanescent
// mode (q real) takes real products, and its q no sine or cosine.  128^2 x 64 FP64: 182 us ->
// 67 us per iteration (0.85 M warp instructions on the FP64 pipe, 43 us at its rate).
constexpr int IG = 8;  // chunks (warps) per block

// a x + y; CPLX false: a is real
template <bool CPLX, typename C> __device__ __forceinline__ C axpy(C a, C x, C y) {
  C r;
  if constexpr (CPLX) {
    r.x = a.x * x.x + (y.x - a.y * x.y);
    r.y = a.x * x.y + (y.y + a.y * x.x);
  } else {
    r.x = a.x * x.x + y.x;
    r.y = a.x * x.y + y.y;
  }
  return r;
}

// One warp's chunk (planes l0 .. l1 - 1, v its V~, overwritten); fe, he, qs as in the kernel.  Returns the
// lane's share of ||U~_{n+1} - U~_n||^2.  Called by every warp of the block (it holds barriers).
template <typename R, bool STEP, int CP, bool CPLX>
__device__ __forceinline__ double interior_chunk(const Problem& P, const cx<R>* __restrict__ vt, cx<R>* v, cx<R> q, cx<R> qc, cx<R> (*fe)[32],
                                                 cx<R> (*he)[32], int l0, int l1, long long nu, bool valid, bool prop,
                                                 R gr, cx<R>* __restrict__ ut, const cx<R>* __restrict__ u0t,
                                                 const cx<R>* __restrict__ inc) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long N2 = (long long)P.n * P.n;
  cx<R> f = czero<R>(), h = czero<R>();
#pragma unroll
  for (int j = 0; j < CP; ++j) {
    if (l0 + j < l1) f = axpy<CPLX>(q, f, v[j]);
    const int jr = CP - 1 - j;
    if (l0 + jr < l1) h = axpy<CPLX>(q, h, v[jr]);
  }
  fe[w][lane] = f;
  he[w][lane] = h;
  __syncthreads();
  // F of the plane before the chunk (every chunk before it is full) and H of the plane after
  // it (the last chunk that holds planes may be short, and no chunk follows it)
  f = czero<R>();
  h = czero<R>();
  for (int c = 0; c < w; ++c) f = axpy<CPLX>(qc, f, fe[c][lane]);
  for (int c = IG - 1; c > w; --c) h = axpy<CPLX>(qc, h, he[c][lane]);
  double d2 = 0.0;
  if (valid && l0 < l1) {
    // F in place of V~, which is read again below (registers for another block per SM)
#pragma unroll
    for (int j = 0; j < CP; ++j) {
      if (l0 + j < l1) f = axpy<CPLX>(q, f, v[j]);
      v[j] = f;
    }
#pragma unroll
    for (int j = CP - 1; j >= 0; --j) {
      const int l = l0 + j;
      if (l < l1) {
        const cx<R> t = axpy<CPLX>(q, h, v[j]);
        cx<R> un = CPLX && prop ? mk<R>(-gr * t.y, gr * t.x) : mk<R>(gr * t.x, gr * t.y);  // gamma = i g or g
        if (STEP && u0t) {
          un = un + u0t[l * N2 + nu];
        } else if (STEP && CPLX && nu == 0) {  // mode 0 propagates
          un = un + inc[l];
        }
        if (STEP) {
          const cx<R> d = un - ut[l * N2 + nu];
          d2 += (double)d.x * (double)d.x + (double)d.y * (double)d.y;
        }
        ut[l * N2 + nu] = un;
        h = axpy<CPLX>(q, h, vt[l * N2 + nu]);
      }
    }
  }
  return d2;
}

template <typename R, bool STEP, int CP>
__global__ void __launch_bounds__(32 * IG, CP <= 8 ? 3 : 1)
k_interior(Problem P, const cx<R>* __restrict__ vt, cx<R>* __restrict__ ut, double* __restrict__ partial,
           const cx<R>* __restrict__ u0t, const cx<R>* __restrict__ inc) {
  __shared__ cx<R> fe[IG][32], he[IG][32];  // chunk c: F of its last plane and H of its first, from zero
  __shared__ cx<R> qs[2][32];               // q and q^CP
  __shared__ R gs[32];                      // |gamma| with its sign
  __shared__ double red[IG];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int N = P.n, M = P.m;
  const long long N2 = (long long)N * N;
  const long long nu = blockIdx.x * 32LL + lane;
  const bool valid = nu < N2;
  const int i2 = (int)(nu / N), i1 = (int)(nu - (long long)i2 * N);
  const int m1 = i1 < N / 2 ? i1 : i1 - N, m2 = i2 < N / 2 ? i2 : i2 - N;
  const int msq = m1 * m1 + m2 * m2;
  const bool off = !valid || (msq >= P.graz_lo[0] && msq <= P.graz_hi[0]);  // grazing modes: T_nu = 0
  const double qq = P.k0[0] * P.k0[0] - P.kn * P.kn * (double)msq;
  const bool prop = qq >= 0.0;
  const int l0 = w * CP, l1 = min(M, l0 + CP);  // this warp's planes
  cx<R> v[CP];
#pragma unroll
  for (int j = 0; j < CP; ++j) v[j] = valid && l0 + j < l1 ? vt[(l0 + j) * N2 + nu] : czero<R>();
  if (w < 2) {
    const double r = off ? 0.0 : rsqrt64(fabs(qq)), kz = sqrt_from_rsqrt(fabs(qq), r);
    qs[w][lane] = off ? czero<R>() : from_d<R>(exp_ikz_inline(kz_vec(prop, kz), w ? CP * P.hz : P.hz));
    if (w == 0) gs[lane] = (R)(-P.g0[0] * r);
  }
  __syncthreads();
  const cx<R> q = qs[0][lane], qc = qs[1][lane];
  // the same for every warp of the block: they hold the same modes (the barriers inside)
  const bool cplx = __any_sync(0xffffffffu, valid && prop);
  const double d2 =
      cplx ? interior_chunk<R, STEP, CP, true>(P, vt, v, q, qc, fe, he, l0, l1, nu, valid, prop, gs[lane], ut, u0t, inc)
           : interior_chunk<R, STEP, CP, false>(P, vt, v, q, qc, fe, he, l0, l1, nu, valid, prop, gs[lane], ut, u0t, inc);
  if constexpr (STEP) {
    double t = d2;
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) red[w] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int c = 0; c < IG; ++c) s += red[c];
      partial[blockIdx.x] = s;
    }
  }
}

template <typename R, bool STEP>
cudaError_t launch_interior(const Problem& Q, const cx<R>* vt, cx<R>* ut, double* partial, const cx<R>* u0t,
                            const cx<R>* inc, cudaStream_t s) {
  const unsigned g = (unsigned)(((long long)Q.n * Q.n + 31) / 32);
  if (Q.m <= IG * 2) k_interior<R, STEP, 2><<<g, 32 * IG, 0, s>>>(Q, vt, ut, partial, u0t, inc);
  else if (Q.m <= IG * 4) k_interior<R, STEP, 4><<<g, 32 * IG, 0, s>>>(Q, vt, ut, partial, u0t, inc);
  else if (Q.m <= IG * 8) k_interior<R, STEP, 8><<<g, 32 * IG, 0, s>>>(Q, vt, ut, partial, u0t, inc);
  else k_interior<R, STEP, 16><<<g, 32 * IG, 0, s>>>(Q, vt, ut, partial, u0t, inc);
  return cudaGetLastError();
}

// ---- GMRES on u - omega^2 T(xi u) = u0 (the Krylov fallback) -----------------
constexpr int GM_BLOCKS = 512;  // blocks of the reduction kernels (grid-stride)

// the plane wave u0 = exp(-i k0 z'_l) on X
template <typename R>
__global__ void k_plane_wave(Problem P, cx<R>* __restrict__ u) {
  const long long N2 = (long long)P.n * P.n, count = (long long)P.m * N2;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < count;
       e += (long long)gridDim.x * blockDim.x) {
    const int l = (int)(e / N2);
    double s, c;
    sincos(-P.k0[0] * (P.z1 + (l + 0.5) * P.hz), &s, &c);
    u[e] = from_d<R>(make_double2(c, s));
  }
}

// y <- xi a
template <typename R>
__global__ void k_xi_times(long long count, const R* __restrict__ xi, const cx<R>* __restrict__ a,
                           cx<R>* __restrict__ y) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < count;
       e += (long long)gridDim.x * blockDim.x) {
    const R x = xi[e];
    const cx<R> v = a[e];
    y[e] = mk<R>(x * v.x, x * v.y);
  }
}

// y <- a - b
template <typename R>
__global__ void k_sub(long long count, const cx<R>* __restrict__ a, const cx<R>* __restrict__ b,
                      cx<R>* __restrict__ y) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < count;
       e += (long long)gridDim.x * blockDim.x)
    y[e] = a[e] - b[e];
}

// block partials of <v_i, w> = sum conj(v_i) w (FP64 sums), grid (GM_BLOCKS, nv):
// partial[i * GM_BLOCKS + block]; summed on the host in a fixed order
template <typename R>
__global__ void __launch_bounds__(FP_T)
k_dots(long long count, const cx<R>* __restrict__ V, long long ld, const cx<R>* __restrict__ w,
       double2* __restrict__ partial) {
  __shared__ double2 red[FP_T];
  const cx<R>* v = V + blockIdx.y * ld;
  double2 acc = make_double2(0.0, 0.0);
  for (long long e = blockIdx.x * (long long)FP_T + threadIdx.x; e < count; e += (long long)gridDim.x * FP_T) {
    const double2 a = to_d(v[e]), b = to_d(w[e]);
    acc.x += a.x * b.x + a.y * b.y;
    acc.y += a.x * b.y - a.y * b.x;
  }
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int h = FP_T / 2; h > 0; h >>= 1) {
    if (threadIdx.x < h) red[threadIdx.x] = red[threadIdx.x] + red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.y * gridDim.x + blockIdx.x] = red[0];
}

// w <- w + sign sum_{i < nv} c_i v_i  (c on the device)
template <typename R>
__global__ void k_comb(long long count, const cx<R>* __restrict__ V, long long ld, int nv,
                       const double2* __restrict__ c, double sign, cx<R>* __restrict__ w) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < count;
       e += (long long)gridDim.x * blockDim.x) {
    double2 acc = to_d(w[e]);
    for (int i = 0; i < nv; ++i) {
      const double2 t = c[i] * to_d(V[i * ld + e]);
      acc.x += sign * t.x;
      acc.y += sign * t.y;
    }
    w[e] = from_d<R>(acc);
  }
}

// y <- s x (s real)
template <typename R>
__global__ void k_scale(long long count, const cx<R>* __restrict__ x, double s, cx<R>* __restrict__ y) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < count;
       e += (long long)gridDim.x * blockDim.x) {
    const double2 v = to_d(x[e]);
    y[e] = from_d<R>(make_double2(s * v.x, s * v.y));
  }
}

}  // namespace

namespace {

constexpr int GM_RESTART = 30;  // Krylov vectors per GMRES cycle

template <typename R> struct FwdLayout {
  long long N2, MN2;
  long long vec_elems;
  cx<R>* base;
  explicit FwdLayout(const Problem& P, void* ws) {
    N2 = (long long)P.n * P.n;
    MN2 = (long long)P.m * N2;
    // fixed point: ut, sc, U~0 of a given incident field; GMRES: sc, tv, x, u0,
    // GM_RESTART + 1 Krylov vectors
    const long long fp = 3 * MN2;
    const long long gm = (5 + GM_RESTART) * MN2;
    vec_elems = fp > gm ? fp : gm;
    base = reinterpret_cast<cx<R>*>(ws);
  }
  double2* reals() const { return reinterpret_cast<double2*>(base + vec_elems); }
  static constexpr size_t partial_elems() { return (size_t)(GM_RESTART + 1) * GM_BLOCKS + (GM_RESTART + 1); }
  static constexpr size_t real_elems() { return partial_elems() + 1024; }  // and the incident wave [M]
  static_assert((size_t)MAX_N * MAX_N / 32 <= 2 * ((size_t)(GM_RESTART + 1) * GM_BLOCKS), "block partials of k_interior");
};

template <typename R>
Problem one_frequency(const Problem& P, int om) {
  Problem Q = P;
  Q.n_omega = 1;
  Q.omega[0] = P.omega[om];
  Q.graz_lo[0] = P.graz_lo[om];
  Q.graz_hi[0] = P.graz_hi[om];
  Q.k0[0] = P.k0[om];
  Q.g0[0] = P.g0[om];
  return Q;
}

// ||a||^2 of count complex values: block partials of k_dots summed on the host in a fixed order
template <typename R>
cudaError_t norm2_host(const cx<R>* a, long long count, double2* partial, cudaStream_t s, double* out);

// Algorithm 1 for one frequency.  On convergence U~ is in the workspace's first field, and
// V~ = F_r[xi F^-1 U~] of it in *vt.  The stopping test is taken on the host each iteration,
// but the transform of the next V~, which only reads U~, is enqueued before the host waits for
// the test's value (mapped page-locked `host`, event `ev`): the wait hides behind it, and at
// convergence it is the V~ that eq. (7) needs.  Not so in the last iteration allowed, which mostly ends
// a solve that fails.  Without convergence nothing is left running on return: xi is the caller's again.
template <typename R>
cudaError_t fixed_point_one(const Problem& Q, const R* xi, const cx<R>* u0, const FwdLayout<R>& L, const cx<R>* tw,
                            double rtol, int max_iter, cudaStream_t s, volatile double* host, cudaEvent_t ev,
                            cx<R>** vt, int* iters, bool* conv) {
  const long long N2 = L.N2, MN2 = L.MN2;
  cx<R>* ut = L.base;
  cx<R>* sc = ut + MN2;
  cx<R>* u0t = u0 ? sc + MN2 : nullptr;  // U~0 of the given incident field
  double* partial = reinterpret_cast<double*>(L.reals());
  cx<R>* inc = reinterpret_cast<cx<R>*>(L.reals() + FwdLayout<R>::partial_elems());  // M values
  const int nblk = (int)((N2 + 31) / 32);
  double nrm0 = (double)N2 * sqrt((double)Q.m);  // ||U~0||: N^2 |e^{-i k0 z}| on M planes (plane wave)
  cudaError_t e;
  if (u0) {  // U~1 = U~0 = F_r[u0], and its norm for the stopping rule
    if ((e = launch_fft2_dense<R>(u0, u0t, Q.n, Q.m, false, tw, s)) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(ut, u0t, sizeof(cx<R>) * MN2, cudaMemcpyDeviceToDevice, s)) != cudaSuccess) return e;
    if ((e = norm2_host<R>(u0t, MN2, L.reals(), s, &nrm0)) != cudaSuccess) return e;
    nrm0 = sqrt(nrm0);
  } else {
    if ((e = cudaMemsetAsync(ut, 0, sizeof(cx<R>) * MN2, s)) != cudaSuccess) return e;
    k_incident<R><<<(Q.m + 63) / 64, 64, 0, s>>>(Q, ut, inc);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  if ((e = launch_xi_transform<R>(ut, sc, xi, Q.n, Q.m, tw, s)) != cudaSuccess) return e;
  int it = 0;
  bool ok = max_iter == 0;
  while (it < max_iter) {
    ++it;
    if ((e = launch_interior<R, true>(Q, sc, ut, partial, u0t, inc, s)) != cudaSuccess) return e;
    k_sum_partials<<<1, 256, 0, s>>>(partial, nblk, const_cast<double*>(host));
    if ((e = cudaEventRecord(ev, s)) != cudaSuccess) return e;
    const bool ahead = it < max_iter;
    if (ahead && (e = launch_xi_transform<R>(ut, sc, xi, Q.n, Q.m, tw, s)) != cudaSuccess) return e;
    if ((e = cudaEventSynchronize(ev)) != cudaSuccess) return e;
    const double diff = sqrt(*host);
    if (diff <= rtol * nrm0) {
      ok = true;
      if (!ahead && (e = launch_xi_transform<R>(ut, sc, xi, Q.n, Q.m, tw, s)) != cudaSuccess) return e;
      break;
    }
    if (!(diff <= 1e30 * nrm0)) break;  // diverged (or not finite)
  }
  *iters = it;
  *conv = ok;
  *vt = sc;
  return ok ? cudaSuccess : cudaStreamSynchronize(s);
}

template <typename R> struct Krylov {
  const Problem& Q;
  const R* xi;
  const cx<R>* tw;
  cudaStream_t s;
  long long N2, MN2;
  unsigned gx;
  cx<R> *sc, *tv;
  double2* partial;  // (GM_RESTART + 1) * GM_BLOCKS
  double2* coef;     // GM_RESTART + 1
  std::vector<double2> host;

  // y <- x - omega^2 F^-1 T_nu F_r[xi x]
  cudaError_t apply(const cx<R>* x, cx<R>* y) {
    k_xi_times<R><<<gx, FP_T, 0, s>>>(MN2, xi, x, sc);
    cudaError_t e = launch_fft2_dense<R>(sc, sc, Q.n, Q.m, false, tw, s);
    if (e != cudaSuccess) return e;
    if ((e = launch_interior<R, false>(Q, sc, tv, nullptr, nullptr, nullptr, s)) != cudaSuccess) return e;
    if ((e = launch_fft2_dense<R>(tv, tv, Q.n, Q.m, true, tw, s)) != cudaSuccess) return e;
    k_sub<R><<<gx, FP_T, 0, s>>>(MN2, x, tv, y);
    return cudaGetLastError();
  }
  // <v_i, w> for the nv vectors v_i = V + i MN2, summed on the host in a fixed order
  cudaError_t dots(const cx<R>* V, int nv, const cx<R>* w, std::vector<std::complex<double>>& out) {
    k_dots<R><<<dim3(GM_BLOCKS, nv), FP_T, 0, s>>>(MN2, V, MN2, w, partial);
    host.resize((size_t)nv * GM_BLOCKS);
    cudaError_t e = cudaMemcpyAsync(host.data(), partial, sizeof(double2) * host.size(), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) return e;
    out.assign(nv, 0.0);
    for (int i = 0; i < nv; ++i) {
      double re = 0.0, im = 0.0;
      for (int b = 0; b < GM_BLOCKS; ++b) {
        re += host[(size_t)i * GM_BLOCKS + b].x;
        im += host[(size_t)i * GM_BLOCKS + b].y;
      }
      out[i] = std::complex<double>(re, im);
    }
    return cudaSuccess;
  }
  // w <- w + sign sum_i c_i v_i
  cudaError_t comb(const cx<R>* V, const std::vector<std::complex<double>>& c, double sign, cx<R>* w) {
    std::vector<double2> ch(c.size());
    for (size_t i = 0; i < c.size(); ++i) ch[i] = make_double2(c[i].real(), c[i].imag());
    cudaError_t e = cudaMemcpyAsync(coef, ch.data(), sizeof(double2) * ch.size(), cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    k_comb<R><<<gx, FP_T, 0, s>>>(MN2, V, MN2, (int)c.size(), coef, sign, w);
    // the host vector must outlive the copy
    return cudaStreamSynchronize(s);
  }
};

// Restarted GMRES(GM_RESTART) with classical Gram-Schmidt applied twice and Givens
// rotations, from x = 0, to ||u0 - A x|| <= rtol ||u0|| (the residual of each cycle's
// start is computed, not estimated); iters counts the operator applications.
template <typename R>
cudaError_t norm2_host(const cx<R>* a, long long count, double2* partial, cudaStream_t s, double* out) {
  k_dots<R><<<dim3(GM_BLOCKS, 1), FP_T, 0, s>>>(count, a, count, a, partial);
  cudaError_t e = cudaGetLastError();
  std::vector<double2> h(GM_BLOCKS);
  if (e == cudaSuccess) e = cudaMemcpyAsync(h.data(), partial, sizeof(double2) * GM_BLOCKS, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return e;
  double t = 0.0;
  for (int b = 0; b < GM_BLOCKS; ++b) t += h[b].x;
  *out = t;
  return cudaSuccess;
}

template <typename R>
cudaError_t gmres_one(const Problem& Q, const R* xi, const cx<R>* u0, const FwdLayout<R>& L, const cx<R>* tw,
                      double rtol, int max_iter, cudaStream_t s, cx<R>** uo, int* iters, bool* conv) {
  using cd = std::complex<double>;
  const long long N2 = L.N2, MN2 = L.MN2;
  Krylov<R> K{Q, xi, tw, s};
  K.N2 = N2;
  K.MN2 = MN2;
  K.gx = (unsigned)((MN2 + FP_T - 1) / FP_T < 4096 ? (MN2 + FP_T - 1) / FP_T : 4096);
  K.sc = L.base;
  K.tv = K.sc + MN2;
  cx<R>* x = K.tv + MN2;
  cx<R>* bv = x + MN2;
  cx<R>* V = bv + MN2;
  K.partial = L.reals();
  K.coef = K.partial + (size_t)(GM_RESTART + 1) * GM_BLOCKS;
  cudaError_t e;
  if (u0) {
    if ((e = cudaMemcpyAsync(bv, u0, sizeof(cx<R>) * MN2, cudaMemcpyDeviceToDevice, s)) != cudaSuccess) return e;
  } else {
    k_plane_wave<R><<<K.gx, FP_T, 0, s>>>(Q, bv);
  }
  if ((e = cudaMemsetAsync(x, 0, sizeof(cx<R>) * MN2, s)) != cudaSuccess) return e;
  std::vector<cd> d;
  if ((e = K.dots(bv, 1, bv, d)) != cudaSuccess) return e;
  const double beta0 = sqrt(d[0].real());
  int total = 0;
  bool ok = false;
  const int R1 = GM_RESTART + 1;
  for (;;) {
    // residual r = u0 - A x in V_0
    if (total == 0) {
      e = cudaMemcpyAsync(V, bv, sizeof(cx<R>) * MN2, cudaMemcpyDeviceToDevice, s);
    } else {
      if ((e = K.apply(x, V)) != cudaSuccess) return e;
      k_sub<R><<<K.gx, FP_T, 0, s>>>(MN2, bv, V, V);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) return e;
    if ((e = K.dots(V, 1, V, d)) != cudaSuccess) return e;
    const double beta = sqrt(d[0].real());
    if (beta <= rtol * beta0) {
      ok = true;
      break;
    }
    if (total >= max_iter || !(beta <= 1e30 * beta0)) break;
    k_scale<R><<<K.gx, FP_T, 0, s>>>(MN2, V, 1.0 / beta, V);
    std::vector<cd> H((size_t)R1 * GM_RESTART, 0.0), g(R1, 0.0), sn(GM_RESTART, 0.0);
    std::vector<double> cs(GM_RESTART, 0.0);
    auto h = [&](int i, int j) -> cd& { return H[(size_t)i * GM_RESTART + j]; };
    g[0] = beta;
    int k = 0;
    for (int j = 0; j < GM_RESTART && total < max_iter; ++j) {
      cx<R>* w = V + (long long)(j + 1) * MN2;
      if ((e = K.apply(V + (long long)j * MN2, w)) != cudaSuccess) return e;
      ++total;
      for (int pass = 0; pass < 2; ++pass) {  // w -= V (V^H w), twice
        if ((e = K.dots(V, j + 1, w, d)) != cudaSuccess) return e;
        if ((e = K.comb(V, d, -1.0, w)) != cudaSuccess) return e;
        for (int i = 0; i <= j; ++i) h(i, j) += d[i];
      }
      if ((e = K.dots(w, 1, w, d)) != cudaSuccess) return e;
      const double hn = sqrt(d[0].real());
      h(j + 1, j) = hn;
      for (int i = 0; i < j; ++i) {  // earlier rotations on column j
        const cd t = cs[i] * h(i, j) + sn[i] * h(i + 1, j);
        h(i + 1, j) = -std::conj(sn[i]) * h(i, j) + cs[i] * h(i + 1, j);
        h(i, j) = t;
      }
      const cd a = h(j, j);
      const double r = std::sqrt(std::norm(a) + hn * hn);
      if (std::abs(a) == 0.0) {
        cs[j] = 0.0;
        sn[j] = 1.0;
      } else {
        cs[j] = std::abs(a) / r;
        sn[j] = (a / std::abs(a)) * hn / r;
      }
      h(j, j) = cs[j] * a + sn[j] * hn;
      h(j + 1, j) = 0.0;
      g[j + 1] = -std::conj(sn[j]) * g[j];
      g[j] = cs[j] * g[j];
      k = j + 1;
      if (!(hn > 0.0) || std::abs(g[j + 1]) <= rtol * beta0) break;
      k_scale<R><<<K.gx, FP_T, 0, s>>>(MN2, w, 1.0 / hn, w);
    }
    std::vector<cd> y(k);
    for (int i = k - 1; i >= 0; --i) {  // H y = g, upper triangular
      cd t = g[i];
      for (int c = i + 1; c < k; ++c) t -= h(i, c) * y[c];
      y[i] = h(i, i) != 0.0 ? t / h(i, i) : cd(0.0);  // (an exactly singular H: a lucky breakdown)
    }
    if (k > 0 && (e = K.comb(V, y, 1.0, x)) != cudaSuccess) return e;
  }
  *iters = total;
  *conv = ok;
  *uo = x;
  return cudaSuccess;
}

}  // namespace

template <typename R>
size_t forward_bytes(const Problem& P) {
  FwdLayout<R> L(P, nullptr);
  return sizeof(cx<R>) * (size_t)L.vec_elems + sizeof(double2) * FwdLayout<R>::real_elems() + 256;
}

template <typename R>
cudaError_t forward_solve(const Problem& P, const R* xi, const cx<R>* incident, cx<R>* W, cx<R>* u_out, void* ws,
                          int method, double rtol, int max_iter, const cx<R>* tw, cudaStream_t s, double* host,
                          cudaEvent_t ev, int* iters, int* converged) {
  const FwdLayout<R> L(P, ws);
  const long long N2 = L.N2, MN2 = L.MN2;
  const unsigned gx = (unsigned)((MN2 + FP_T - 1) / FP_T < 4096 ? (MN2 + FP_T - 1) / FP_T : 4096);
  cudaError_t e = cudaSuccess;
  for (int om = 0; om < P.n_omega; ++om) {
    const Problem Q = one_frequency<R>(P, om);
    cx<R>* uo_user = u_out ? u_out + (long long)om * MN2 : nullptr;
    cx<R>* vt = nullptr;  // V~ of the converged field
    int it = 0;
    bool conv = false;
    const cx<R>* u0 = incident ? incident + (long long)om * MN2 : nullptr;
    if (method != 1) {  // Algorithm 1 (method 0, or the first try of method 2)
      if ((e = fixed_point_one<R>(Q, xi, u0, L, tw, rtol, max_iter, s, host, ev, &vt, &it, &conv)) != cudaSuccess)
        return e;
      if (conv && uo_user && (e = launch_fft2_dense<R>(L.base, uo_user, P.n, P.m, true, tw, s)) != cudaSuccess)
        return e;  // u = F^-1 U~
    }
    if (!conv && method != 0) {  // GMRES (method 1, or the fallback of method 2)
      int it2 = 0;
      cx<R>* u = nullptr;
      if ((e = gmres_one<R>(Q, xi, u0, L, tw, rtol, max_iter, s, &u, &it2, &conv)) != cudaSuccess) return e;
      it += it2;
      if (conv) {
        if (uo_user &&
            (e = cudaMemcpyAsync(uo_user, u, sizeof(cx<R>) * MN2, cudaMemcpyDeviceToDevice, s)) != cudaSuccess)
          return e;
        vt = L.base;  // the Krylov scratch: u lies behind it
        k_xi_times<R><<<gx, FP_T, 0, s>>>(MN2, xi, u, vt);
        if ((e = launch_fft2_dense<R>(vt, vt, P.n, P.m, false, tw, s)) != cudaSuccess) return e;
      }
    }
    if (iters) iters[om] = it;
    if (converged) converged[om] = conv ? 1 : 0;
    if (!conv) return cudaSuccess;
    // eq. (7) with the converged field
    cx<R>* wo = W + (long long)om * P.m1 * N2;
    if ((e = launch_apply_data<R>(Q, vt, false, wo, s)) != cudaSuccess) return e;
    if ((e = launch_fft2_dense<R>(wo, wo, P.n, P.m1, true, tw, s)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template size_t forward_bytes<double>(const Problem&);
template size_t forward_bytes<float>(const Problem&);
template cudaError_t forward_solve<double>(const Problem&, const double*, const double2*, double2*, double2*, void*,
                                           int, double, int, const double2*, cudaStream_t, double*, cudaEvent_t, int*,
                                           int*);
template cudaError_t forward_solve<float>(const Problem&, const float*, const float2*, float2*, float2*, void*, int,
                                          double, int, const float2*, cudaStream_t, double*, cudaEvent_t, int*, int*);

}  // namespace fl
