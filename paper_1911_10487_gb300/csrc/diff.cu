// Derivatives of the reconstruction at a fixed Tikhonov parameter alpha_omega
// per frequency (Algorithm 2, Sec. 4, without the discrepancy search):
//
//   (W, log alpha) -> (xi, Phi),   Phi_omega = sum_nu ||A_nu V~_nu - W~_nu||^2.
//
// Every data plane lies above X, so the matrix of eq. (8) is exactly rank one,
// A_kl = E_k P_l with E_k = gamma e^{i k_z (z_k - z_top)}, P_l = e^{i k_z (z_top - z'_l)}
// (solve_rank1.cu), and (A A^H + alpha I)^-1 needs no matrix at all.  With e = E / ||E||,
// tr = ||E||^2 ||P||^2, mu = tr / (tr + alpha), kappa = alpha / (tr + alpha),
// eta = ||E|| / (tr + alpha) and c = e^H b:
//
//   V~_l = conj(P_l) eta c                    (= A^H (A A^H + alpha I)^-1 b)
//   U~_l = U~0_l + T_l V~_l                   eq. (9): V~ is a power of q = e^{i k_z h_z}
//                                             along the planes, so its two recurrences sum
//                                             to the factor T_l of the geometry,
//       evanescent (q real):  T_l = gamma (sum_{j <= l} q^2j + (M - 1 - l))
//       propagating (|q| = 1): T_l = gamma ((l + 1) + sum_{1 <= j <= M-1-l} q^2j)
//   Phi  = ||g||^2 + kappa^2 mu (1 + kappa) |c|^2,  g = b - mu (1 + kappa) c e
// then V = F^-1[V~], u = F^-1[U~] and xi = Re(sum conj(u) V) / sum |u|^2 (step 3).
//   VJP:  tau = sum_l P_l (V~-bar_l + conj(T_l) U~-bar_l)
//         b-bar = eta tau e + 2 Phi-bar g       (g is half the gradient of Phi in b)
//         lnalpha-bar = -kappa Re(conj(tau) eta c) + 2 Phi-bar kappa^2 mu |c|^2
//   JVP:  c-dot = e^H b-dot,  V~-dot_l = conj(P_l) eta (c-dot - kappa lnalpha-dot c),
//         U~-dot_l = T_l V~-dot_l,
//         Phi-dot = 2 Re g^H b-dot + 2 kappa^2 mu lnalpha-dot |c|^2
// The tape keeps c and g per mode.  Modes with no solution (grazing, a matrix that
// underflowed, or alpha / tr beyond AP_MAX where V~ is zero in FP64) are mu = eta = 0,
// kappa = 1: V~ = 0 and g = b, their residual.  Gradients use grad z = dL/dRe z + i dL/dIm z.
//
// What bounds it.  A dense factorisation costs ~(4/3) M1^3 FP64 operations per mode, and
// all N^2 modes are solved at a fixed alpha; the closed form is O(M1 + M) per mode, and the
// kernels stream their fields (128^2 x 64, 32 data planes, 4 frequencies, mixed precision;
// Cholesky factors before, this form now): forward 16.6 ms -> 58 us for 150 MB, VJP 8.6 ms ->
// 95 us for 170 MB, 16 JVP directions 107.8 ms -> 480-495 us for 1.4 GB (565 us with four directions per pass over
// the planes instead of eight).  A block holds 32 consecutive modes (lanes: every access to a plane
// is one 256-byte row) and splits the data planes and blocks of PB X planes
// over its DG warps, so that a small grid still fills the SMs.  The geometry (e, q, gamma, and
// P and T at one plane of each block of PB) is tabulated once per plan in FP64; inside a block
// of planes P and T follow by at most PB - 1 products, whose rounding is that of the
// exponentials themselves.  FS_FP64 computes in FP64, FS_MIXED in two-float arithmetic
// (~48 bits, twofloat.cuh) on the FP32 pipe from tables split into two floats: on this GPU
// FP64 instructions and conversions run at 1/64 of the FP32 rate, and the fields in and out
// are FP32.
// Per-frequency sums (Phi, lnalpha-bar, Phi-dot) go to per-block partials reduced in a fixed
// order, so results do not depend on scheduling.
#include <math.h>

#include "diff.cuh"
#include "modes.cuh"
#include "twofloat.cuh"

namespace fl {

namespace {

constexpr int PB = DIFF_PB;       // X planes per block of planes
constexpr int DG = 8;             // warps per block
constexpr int DT = 32 * DG;       // threads per block of the per-mode kernels
constexpr int KC = DENSE_M1 / DG; // data planes per warp
constexpr int JG = 8;             // JVP directions per pass over the planes
constexpr double AP_MAX = 1e290;  // alpha / tr above this: V~ = 0 in FP64
static_assert(DENSE_M <= PB * DG, "one block of planes per warp");
static_assert(DENSE_M1 == KC * DG, "data planes dealt over the warps");

// The arithmetic of the per-mode kernels: FP64, or two-float in the mixed precision.
template <typename R> struct Wide;
template <> struct Wide<double> {
  using T = double;   // value
  using S = double;   // one component in a table
  using SC = double2; // a complex value on the tape
  __device__ __forceinline__ static T ld(const S* p) { return *p; }
  __device__ __forceinline__ static S st(double x) { return x; }
  __device__ __forceinline__ static T from(double x) { return x; }
  __device__ __forceinline__ static T from_r(double x) { return x; }
  __device__ __forceinline__ static double d(T x) { return x; }
  __device__ __forceinline__ static double r(T x) { return x; }
  __device__ __forceinline__ static T neg(T a) { return -a; }
  __device__ __forceinline__ static T add(T a, T b) { return a + b; }
  __device__ __forceinline__ static T mul(T a, T b) { return a * b; }
  __device__ __forceinline__ static T mulr(T a, double x) { return a * x; }
  __device__ __forceinline__ static T fma(T a, T b, T c) { return a * b + c; }
  __device__ __forceinline__ static T fmar(T a, double x, T c) { return a * x + c; }
  __device__ __forceinline__ static T wsum(T a) { return warp_sum(a); }
  using Acc = double;  // a running sum of products
  __device__ __forceinline__ static void mac(Acc& s, T a, double x) { s = a * x + s; }
  __device__ __forceinline__ static T sum(Acc s) { return s; }
  __device__ __forceinline__ static double mulround(T a, T b) { return a * b; }
  __device__ __forceinline__ static SC pack(T re, T im) { return make_double2(re, im); }
  __device__ __forceinline__ static void unpack(SC v, T& re, T& im) { re = v.x; im = v.y; }
};
template <> struct Wide<float> {
  using T = ff;
  using S = float2;
  using SC = float4;
  __device__ __forceinline__ static T ld(const S* p) { const float2 v = *p; return ff{v.x, v.y}; }
  __device__ __forceinline__ static S st(double x) { const ff v = ff_from(x); return make_float2(v.hi, v.lo); }
  __device__ __forceinline__ static T from(double x) { return ff_from(x); }
  __device__ __forceinline__ static T from_r(float x) { return ff{x, 0.f}; }
  __device__ __forceinline__ static double d(T x) { return ff_to(x); }
  __device__ __forceinline__ static float r(T x) { return x.hi + x.lo; }
  __device__ __forceinline__ static T neg(T a) { return ff_neg(a); }
  __device__ __forceinline__ static T add(T a, T b) { return ff_add(a, b); }
  __device__ __forceinline__ static T mul(T a, T b) { return ff_mul(a, b); }
  __device__ __forceinline__ static T mulr(T a, float x) { return ff_mul_f(a, x); }
  __device__ __forceinline__ static T fma(T a, T b, T c) { return ff_add(ff_mul(a, b), c); }
  __device__ __forceinline__ static T fmar(T a, float x, T c) { return ff_add(ff_mul_f(a, x), c); }
  __device__ __forceinline__ static T wsum(T a) { return ff_warp_sum(a); }
  // compensated sums (Dot2, twofloat.cuh): two thirds of the operations of two-float sums
  using Acc = dot2;
  __device__ __forceinline__ static void mac(Acc& s, T a, float x) {
    const float p = a.hi * x;
    dot2_add(s, p, fmaf(a.lo, x, fmaf(a.hi, x, -p)));
  }
  __device__ __forceinline__ static T sum(Acc s) { return fast_two_sum(s.s, s.e); }
  // the product rounded to FP32
  __device__ __forceinline__ static float mulround(T a, T b) {
    const float p = a.hi * b.hi;
    return p + fmaf(a.lo, b.hi, fmaf(a.hi, b.lo, fmaf(a.hi, b.hi, -p)));
  }
  __device__ __forceinline__ static SC pack(T re, T im) { return make_float4(re.hi, re.lo, im.hi, im.lo); }
  __device__ __forceinline__ static void unpack(SC v, T& re, T& im) { re = ff{v.x, v.y}; im = ff{v.z, v.w}; }
};

template <typename T> struct WC { T re, im; };  // complex value

__device__ __forceinline__ int exponent_of(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7ff) - 1023; }
__device__ __forceinline__ int exponent_of(float x) { return (int)((__float_as_int(x) >> 23) & 0xff) - 127; }

// A complex factor that multiplies wide values into outputs.  Two-float holds it as a
// mantissa and a power of two: FP64 reaches factors (eta c, 2 Phi-bar N^2) outside the FP32
// range whose products with the fields are inside it.  (The power goes to 2^+-126; a mantissa
// takes the rest, to 2^252.)
template <typename R> struct Factor;
template <> struct Factor<double> {
  double re, im;
  __device__ __forceinline__ static Factor make(double2 v) { return Factor{v.x, v.y}; }
  __device__ __forceinline__ double out(double x) const { return x; }
};
template <> struct Factor<float> {
  ff re, im;
  float s;
  __device__ __forceinline__ static Factor make(double2 v) {
    const double a = fmax(fabs(v.x), fabs(v.y));
    int e = 0;
    if (a > 0.0 && isfinite(a)) e = exponent_of(a);
    e = e < -126 ? -126 : (e > 126 ? 126 : e);
    const double sc = __longlong_as_double((long long)(1023 - e) << 52);
    Factor f;
    f.re = ff_from(v.x * sc);
    f.im = ff_from(v.y * sc);
    f.s = __int_as_float((e + 127) << 23);
    return f;
  }
  __device__ __forceinline__ float out(ff x) const { return (x.hi + x.lo) * s; }
  __device__ __forceinline__ float out(float x) const { return x * s; }
};

// exponent of the largest of the warp's values (uniform; 0 for all zero): sums of squares
// and products are taken of values scaled by its power of two, which keeps them in the
// FP32 range of the two-float form.  FP64 needs none.
__device__ __forceinline__ int warp_exponent(float a) {
  for (int o = 16; o > 0; o >>= 1) a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, o));
  const int e = exponent_of(a);
  return a > 0.f ? (e < -120 ? -120 : (e > 120 ? 120 : e)) : 0;
}
__device__ __forceinline__ int warp_exponent(double) { return 0; }
__device__ __forceinline__ double scale_by(double x, int) { return x; }
__device__ __forceinline__ ff scale_by(ff x, int e) {
  const float s = __int_as_float((e + 127) << 23);
  return ff{x.hi * s, x.lo * s};
}
__device__ __forceinline__ float scale_by(float x, int e) { return x * __int_as_float((e + 127) << 23); }
__device__ __forceinline__ double pow2d(int e) { return __longlong_as_double((long long)(1023 + e) << 52); }

// ---------------------------------------------------------------------------
// tables of the geometry, one block per 32 modes (k_diff_tables, once per plan), FP64
// ---------------------------------------------------------------------------
struct ModeK {
  double2 kz, gamma;
  bool prop, grazing;
};
__device__ __forceinline__ ModeK mode_k(const Problem& P, int om, long long nu) {
  const int N = P.n;
  const int i2 = (int)(nu / N), i1 = (int)(nu - (long long)i2 * N);
  const int m1 = i1 < N / 2 ? i1 : i1 - N, m2 = i2 < N / 2 ? i2 : i2 - N;
  const int msq = m1 * m1 + m2 * m2;
  ModeK g;
  g.grazing = msq >= P.graz_lo[om] && msq <= P.graz_hi[om];
  const double qq = P.k0[om] * P.k0[om] - P.kn * P.kn * (double)msq;
  g.prop = qq >= 0.0;
  const double kz = g.grazing ? 1.0 : sqrt(fabs(qq));  // k_z = 0 is excluded: a placeholder
  g.kz = g.prop ? make_double2(kz, 0.0) : make_double2(0.0, kz);
  const double gm = g.grazing ? 0.0 : -P.g0[om] / kz;
  g.gamma = g.prop ? make_double2(0.0, gm) : make_double2(gm, 0.0);
  return g;
}

template <typename R>
__global__ void __launch_bounds__(DT) k_diff_tables(Problem P, DiffTables<R> tab, DiffTablesOut<R> out) {
  using W = Wide<R>;
  __shared__ double2 p2[DENSE_M][32];  // |P_l|^2 (evanescent) or P_l^2 (propagating)
  __shared__ double es[DG][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int om = blockIdx.y, n = P.m1, m = P.m;
  const long long N2 = (long long)P.n * P.n;
  const long long nu = (long long)blockIdx.x * 32 + lane;
  const bool valid = nu < N2;
  const ModeK g = mode_k(P, om, valid ? nu : 0);
  const double ztop = P.z1 + (m - 0.5) * P.hz;
  // E_k: an evanescent E is scaled by e^{k_z (z_min - z_top)}, so that its direction e keeps
  // full precision where ||E|| underflows
  const double base = g.prop ? ztop : P.zy_min;
  double2 e[KC];
  double se = 0.0;
#pragma unroll
  for (int i = 0; i < KC; ++i) {
    const int k = w + DG * i;
    e[i] = k < n ? g.gamma * exp_ikz(g.kz, P.zy[k] - base) : make_double2(0.0, 0.0);
    se += abs2(e[i]);
  }
  es[w][lane] = se;
  for (int l = w; l < m; l += DG) {
    const double2 p = exp_ikz(g.kz, ztop - (P.z1 + (l + 0.5) * P.hz));
    p2[l][lane] = g.prop ? p * p : make_double2(abs2(p), 0.0);
    const int a = l / PB, top = min(PB * a + PB, m) - 1;
    if (l == top && valid) {
      const long long at = ((long long)om * tab.nb + a) * N2 + nu;
      out.pr[at] = W::st(p.x);
      out.pi[at] = W::st(p.y);
    }
  }
  __syncthreads();
  double nn = 0.0;
  for (int i = 0; i < DG; ++i) nn += es[i][lane];  // ||E||^2, scaled
  const double rn = nn > 0.0 ? 1.0 / sqrt(nn) : 0.0;
  if (valid)
#pragma unroll
    for (int i = 0; i < KC; ++i) {
      const int k = w + DG * i;
      if (k < n) {
        const long long at = ((long long)om * n + k) * N2 + nu;
        out.er[at] = W::st(rn * e[i].x);
        out.ei[at] = W::st(rn * e[i].y);
      }
    }
  if (w == 0 && valid) {
    const long long at = (long long)om * N2 + nu;
    const double sc = g.prop ? 1.0 : exp(-g.kz.y * (P.zy_min - ztop));
    const double ne = sqrt(nn) * sc;
    const double2 q = exp_ikz(g.kz, P.hz);
    out.q[at] = typename DiffTables<R>::S2{W::st(q.x), W::st(q.y)};
    out.g[at] = W::st(g.prop ? g.gamma.y : g.gamma.x);
    // sums from the top plane down: sum_{j <= l} q^2j = sum |P_{M-1-j}|^2 (evanescent),
    // sum_{1 <= j <= n} q^2j = sum P_{M-1-j}^2 (propagating)
    double2 acc = make_double2(0.0, 0.0);
    for (int j = 0; j < m; ++j) {
      // evanescent: acc = sum_{i <= j} q^2i belongs to plane j, stored at block starts
      // propagating: acc = sum_{1 <= i <= j} q^2i belongs to plane M-1-j, stored at block tops
      if (!g.prop || j > 0) acc = acc + p2[m - 1 - j][lane];
      const int l = g.prop ? m - 1 - j : j, a = l / PB;
      if (g.prop ? l == min(PB * a + PB, m) - 1 : l == PB * a) {
        const double2 s = g.gamma * acc;
        const long long ab = ((long long)om * tab.nb + a) * N2 + nu;
        out.sr[ab] = W::st(s.x);
        out.si[ab] = W::st(s.y);
      }
    }
    const double sp = g.prop ? (double)m : acc.x;  // ||P||^2
    const double tr = g.grazing ? 0.0 : ne * ne * sp;
    out.tr[at] = tr;
    out.ne[at] = tr > 0.0 ? (g.prop ? -ne : ne) : (g.prop ? -0.0 : 0.0);  // the sign marks propagating modes
  }
}

// incident field of mode 0: U~0_l = N^2 e^{-i k0 z'_l}
__global__ void k_diff_incident(Problem P, double2* __restrict__ inc) {
  const int om = blockIdx.x;
  for (int l = threadIdx.x; l < P.m; l += blockDim.x) {
    double s, c;
    sincos(-P.k0[om] * (P.z1 + (l + 0.5) * P.hz), &s, &c);
    const double n2 = (double)P.n * P.n;
    inc[om * P.m + l] = make_double2(n2 * c, n2 * s);
  }
}

// log alpha -> the tape's log alpha and alpha
__global__ void k_diff_alpha(const double* __restrict__ log_alpha, int F, double* __restrict__ la) {
  const int om = threadIdx.x;
  if (om < F) {
    la[om] = log_alpha[om];
    la[F + om] = exp(log_alpha[om]);
  }
}

// the scalars of one mode at alpha
struct ModeScalars { double eta, mu, kappa; };
__device__ __forceinline__ ModeScalars mode_scalars(double tr, double ne, double alpha) {
  ModeScalars s{0.0, 0.0, 1.0};
  if (tr > 0.0 && alpha < AP_MAX * tr) {
    const double r = rcp64(tr + alpha);
    s.eta = fabs(ne) * r;
    s.mu = tr * r;
    s.kappa = alpha * r;
  }
  return s;
}

// P_l and T_l of the planes of block a, handed to f(l, P, T, l-th index j): real (an
// evanescent mode: P and T real) or complex.
template <typename R, typename F>
__device__ __forceinline__ void planes_real(const DiffTables<R>& tab, long long at, long long ab, int a, int m, F f) {
  using W = Wide<R>;
  using T = typename W::T;
  const T q = W::ld(&tab.q[at].x), g = W::ld(tab.g + at);
  const T q2 = W::mul(q, q);
  const int top = min(PB * a + PB, m) - 1;
  T p[PB];
  T cur = W::ld(tab.pr + ab);
#pragma unroll
  for (int j = PB - 1; j >= 0; --j) {
    const int l = PB * a + j;
    if (l < top) cur = W::mul(cur, q);
    p[j] = cur;
  }
  T h = W::ld(tab.sr + ab);
#pragma unroll
  for (int j = 0; j < PB; ++j) {
    const int l = PB * a + j;
    if (l <= top) f(l, j, p[j], W::fmar(g, (R)(m - 1 - l), h));
    h = W::fma(q2, h, g);
  }
}
template <typename R, typename F>
__device__ __forceinline__ void planes_cplx(const DiffTables<R>& tab, long long at, long long ab, int a, int m,
                                            bool prop, F f) {
  using W = Wide<R>;
  using T = typename W::T;
  using C = WC<T>;
  const T zero = W::from(0.0);
  const C q = C{W::ld(&tab.q[at].x), W::ld(&tab.q[at].y)};
  const T g = W::ld(tab.g + at);
  const C q2 = C{W::fma(q.re, q.re, W::neg(W::mul(q.im, q.im))), W::mulr(W::mul(q.re, q.im), (R)2)};
  const int top = min(PB * a + PB, m) - 1;
  C p = C{W::ld(tab.pr + ab), W::ld(tab.pi + ab)};
  C s = C{W::ld(tab.sr + ab), W::ld(tab.si + ab)};
  if (prop) {  // both from the block's top plane down
#pragma unroll 1
    for (int l = top; l >= PB * a; --l) {
      if (l < top) {
        p = C{W::fma(p.re, q.re, W::neg(W::mul(p.im, q.im))), W::fma(p.re, q.im, W::mul(p.im, q.re))};
        const C t = C{s.re, W::add(s.im, g)};  // gamma = i g
        s = C{W::fma(q2.re, t.re, W::neg(W::mul(q2.im, t.im))), W::fma(q2.re, t.im, W::mul(q2.im, t.re))};
      }
      f(l, p, C{s.re, W::fmar(g, (R)(l + 1), s.im)});
    }
  } else {  // an evanescent mode in a warp that also holds propagating ones
    T pv[PB];
    T cur = p.re;
#pragma unroll
    for (int j = PB - 1; j >= 0; --j) {
      if (PB * a + j < top) cur = W::mul(cur, q.re);
      pv[j] = cur;
    }
    T h = s.re;
#pragma unroll
    for (int j = 0; j < PB; ++j) {
      const int l = PB * a + j;
      if (l <= top) f(l, C{pv[j], zero}, C{W::fmar(g, (R)(m - 1 - l), h), zero});
      h = W::fma(q2.re, h, g);
    }
  }
}

// block sum of one double per warp (lane 0's value) -> partial[slot]
__device__ __forceinline__ void block_partial(double v, double* red, double* partial, long long slot) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) red[warp] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < DG; ++w) s += red[w];
    partial[slot] = s;
  }
}

// ---------------------------------------------------------------------------
// forward: tape <- c, g; V~/U~ planes; block partials of Phi
// ---------------------------------------------------------------------------
template <typename R>
__global__ void __launch_bounds__(DT)
k_diff_forward(Problem P, DiffTables<R> tab, const cx<R>* __restrict__ wt, const double* __restrict__ alpha_arr,
               double2* __restrict__ cs, typename Wide<R>::SC* __restrict__ gs, cx<R>* __restrict__ vt,
               cx<R>* __restrict__ ut, double* __restrict__ partial, unsigned long long* __restrict__ ctr) {
  using W = Wide<R>;
  using T = typename W::T;
  __shared__ WC<T> sc[DG][32];
  __shared__ Factor<R> cv_s[32];
  __shared__ WC<T> f_s[32];
  __shared__ double red[DG];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int om = blockIdx.y, n = P.m1, m = P.m;
  const long long N2 = (long long)P.n * P.n;
  const long long nu = (long long)blockIdx.x * 32 + lane;
  const bool valid = nu < N2;
  const long long at = (long long)om * N2 + (valid ? nu : 0);
  const double ne = tab.ne[at];
  const bool prop = signbit(ne);
  const bool cplx = __any_sync(0xffffffffu, prop);
  const T zero = W::from(0.0);
  cx<R> b[KC];
  WC<T> e[KC];
  typename W::Acc ca{}, cb{};
  R big = R(0);
#pragma unroll
  for (int i = 0; i < KC; ++i) {
    const int k = w + DG * i;
    const long long ak = ((long long)om * n + k) * N2 + nu;
    const bool on = valid && k < n;
    b[i] = on ? wt[ak] : czero<R>();
    e[i].re = on ? W::ld(tab.er + ak) : zero;
    e[i].im = on && cplx ? W::ld(tab.ei + ak) : zero;
    big = fmax(big, fmax(fabs(b[i].x), fabs(b[i].y)));
  }
#pragma unroll
  for (int i = 0; i < KC; ++i) {  // c = e^H b
    W::mac(ca, e[i].re, b[i].x);
    W::mac(cb, e[i].re, b[i].y);
    if (cplx) {
      W::mac(ca, e[i].im, b[i].y);
      W::mac(cb, W::neg(e[i].im), b[i].x);
    }
  }
  WC<T> c = WC<T>{W::sum(ca), W::sum(cb)};
  sc[w][lane] = c;
  __syncthreads();
  double phi = 0.0;
  if (w == 0) {
    for (int i = 1; i < DG; ++i) c = WC<T>{W::add(c.re, sc[i][lane].re), W::add(c.im, sc[i][lane].im)};
    const double tr = tab.tr[at], alpha = alpha_arr[om];
    const ModeScalars s = mode_scalars(tr, ne, alpha);
    const double2 cd = make_double2(W::d(c.re), W::d(c.im));
    const double nu1 = s.mu * (1.0 + s.kappa);  // 1 - kappa^2
    cv_s[lane] = Factor<R>::make(s.eta * cd);
    const double2 fd = nu1 * cd;
    f_s[lane] = WC<T>{W::from(fd.x), W::from(fd.y)};
    if (valid) {
      cs[at] = cd;
      phi = s.kappa * s.kappa * nu1 * abs2(cd);
    }
    phi = warp_sum(phi);
    // alpha = 0 (log alpha = -inf): the regularised matrix is singular
    const bool bad = valid && tr > 0.0 && !(alpha > 0.0) && alpha < AP_MAX;
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicAdd(ctr + C_NONFINITE, 1ull);
  }
  __syncthreads();
  const WC<T> f = f_s[lane];
  const int ex = warp_exponent(big);
  T gg = zero;
#pragma unroll
  for (int i = 0; i < KC; ++i) {  // g = b - (1 - kappa^2) c e, ||g||^2
    const int k = w + DG * i;
    if (k < n) {
      T gr = W::add(W::from_r(b[i].x), W::neg(W::mul(f.re, e[i].re)));
      T gi = W::add(W::from_r(b[i].y), W::neg(W::mul(f.im, e[i].re)));
      if (cplx) {
        gr = W::fma(f.im, e[i].im, gr);
        gi = W::add(gi, W::neg(W::mul(f.re, e[i].im)));
      }
      if (valid) gs[((long long)om * n + k) * N2 + nu] = W::pack(gr, gi);
      const T xr = scale_by(gr, -ex), xi = scale_by(gi, -ex);
      gg = W::fma(xr, xr, gg);
      gg = W::fma(xi, xi, gg);
    }
  }
  gg = W::wsum(gg);
  phi += W::d(gg) * (pow2d(ex) * pow2d(ex));
  const Factor<R> cv = cv_s[lane];
  for (int a = w; a < tab.nb; a += DG) {
    if (!valid) break;
    const long long ab = ((long long)om * tab.nb + a) * N2 + nu;
    const long long o0 = (long long)om * m * N2 + nu;
    const bool inc = nu == 0;
    auto put = [&](int l, T vr, T vi, T ur, T ui) {
      vt[o0 + l * N2] = mk<R>(cv.out(vr), cv.out(vi));
      if (inc) {
        const double2 z = tab.inc[om * m + l];
        ut[o0 + l * N2] = mk<R>((R)((double)cv.out(ur) + z.x), (R)((double)cv.out(ui) + z.y));
      } else {
        ut[o0 + l * N2] = mk<R>(cv.out(ur), cv.out(ui));
      }
    };
    if (!cplx) {
      planes_real<R>(tab, at, ab, a, m, [&](int l, int, T p, T t) {
        const T vr = W::mul(p, cv.re), vi = W::mul(p, cv.im);
        put(l, vr, vi, W::mul(t, vr), W::mul(t, vi));
      });
    } else {
      planes_cplx<R>(tab, at, ab, a, m, prop, [&](int l, WC<T> p, WC<T> t) {
        const T vr = W::fma(p.re, cv.re, W::mul(p.im, cv.im));  // conj(P) c
        const T vi = W::fma(p.re, cv.im, W::neg(W::mul(p.im, cv.re)));
        put(l, vr, vi, W::fma(t.re, vr, W::neg(W::mul(t.im, vi))), W::fma(t.re, vi, W::mul(t.im, vr)));
      });
    }
  }
  block_partial(phi, red, partial, (long long)om * gridDim.x + blockIdx.x);
}

// ---------------------------------------------------------------------------
// VJP: N^2 b-bar per mode (for the inverse transform) and the lnalpha-bar partials.
// vbt/ubt (the forward transforms of V-bar, u-bar; the adjoint of F^-1 is F / N^2) may
// be null when xi carries no cotangent; wbt may be null when W needs no gradient.
// ---------------------------------------------------------------------------
template <typename R>
__global__ void __launch_bounds__(DT)
k_diff_vjp(Problem P, DiffTables<R> tab, const double2* __restrict__ cs, const typename Wide<R>::SC* __restrict__ gs,
           const cx<R>* __restrict__ vbt, const cx<R>* __restrict__ ubt, const double* __restrict__ alpha_arr,
           const double* __restrict__ grad_phi, cx<R>* __restrict__ wbt, double* __restrict__ partial) {
  using W = Wide<R>;
  using T = typename W::T;
  __shared__ WC<T> sc[DG][32];
  __shared__ Factor<R> t_s[32];
  __shared__ Factor<R> gf_s;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int om = blockIdx.y, n = P.m1, m = P.m;
  const long long N2 = (long long)P.n * P.n;
  const long long nu = (long long)blockIdx.x * 32 + lane;
  const bool valid = nu < N2;
  const long long at = (long long)om * N2 + (valid ? nu : 0);
  const double ne = tab.ne[at];
  const bool prop = signbit(ne);
  const bool cplx = __any_sync(0xffffffffu, prop);
  const T zero = W::from(0.0);
  const double gphi = grad_phi ? grad_phi[om] : 0.0;
  T tr_ = zero, ti_ = zero;
  if (vbt && valid) {
    for (int a = w; a < tab.nb; a += DG) {
      const long long ab = ((long long)om * tab.nb + a) * N2 + nu;
      const long long o0 = (long long)om * m * N2 + nu;
      if (!cplx) {
        cx<R> vb[PB], ub[PB];
#pragma unroll
        for (int j = 0; j < PB; ++j) {  // the block's loads in flight together
          const int l = PB * a + j;
          vb[j] = l < m ? vbt[o0 + l * N2] : czero<R>();
          ub[j] = l < m ? ubt[o0 + l * N2] : czero<R>();
        }
        planes_real<R>(tab, at, ab, a, m, [&](int l, int j, T p, T t) {
          tr_ = W::fma(p, W::fmar(t, ub[j].x, W::from_r(vb[j].x)), tr_);
          ti_ = W::fma(p, W::fmar(t, ub[j].y, W::from_r(vb[j].y)), ti_);
        });
      } else {
        planes_cplx<R>(tab, at, ab, a, m, prop, [&](int l, WC<T> p, WC<T> t) {
          const cx<R> v = vbt[o0 + l * N2], u = ubt[o0 + l * N2];
          // V-bar + conj(T) U-bar
          const T xr = W::fmar(t.im, u.y, W::fmar(t.re, u.x, W::from_r(v.x)));
          const T xi = W::fmar(W::neg(t.im), u.x, W::fmar(t.re, u.y, W::from_r(v.y)));
          tr_ = W::add(tr_, W::fma(p.re, xr, W::neg(W::mul(p.im, xi))));
          ti_ = W::add(ti_, W::fma(p.re, xi, W::mul(p.im, xr)));
        });
      }
    }
  }
  sc[w][lane] = WC<T>{tr_, ti_};
  __syncthreads();
  if (w == 0) {
    for (int i = 1; i < DG; ++i) {
      tr_ = W::add(tr_, sc[i][lane].re);
      ti_ = W::add(ti_, sc[i][lane].im);
    }
    const ModeScalars s = mode_scalars(tab.tr[at], ne, alpha_arr[om]);
    const double2 c = cs[at];
    const double2 t = s.eta * make_double2(W::d(tr_), W::d(ti_));  // N^2 eta tau
    t_s[lane] = Factor<R>::make(t);
    double lbar = 0.0;
    if (valid) {
      lbar = -s.kappa * P.inv_n2 * (t.x * c.x + t.y * c.y);
      if (grad_phi) lbar += 2.0 * gphi * s.kappa * s.kappa * s.mu * abs2(c);
    }
    lbar = warp_sum(lbar);
    if (lane == 0) {
      partial[(long long)om * gridDim.x + blockIdx.x] = lbar;
      gf_s = Factor<R>::make(make_double2(2.0 * gphi * (double)N2, 0.0));
    }
  }
  if (!wbt) return;
  __syncthreads();
  const Factor<R> t = t_s[lane], gf = gf_s;
#pragma unroll
  for (int i = 0; i < KC; ++i) {
    const int k = w + DG * i;
    if (valid && k < n) {
      const long long ak = ((long long)om * n + k) * N2 + nu;
      R br = R(0), bi = R(0);
      const T er = W::ld(tab.er + ak), ei = cplx ? W::ld(tab.ei + ak) : zero;
      T xr = W::mul(er, t.re), xi = W::mul(er, t.im);
      if (cplx) {
        xr = W::add(xr, W::neg(W::mul(ei, t.im)));
        xi = W::fma(ei, t.re, xi);
      }
      br = t.out(xr);
      bi = t.out(xi);
      if (grad_phi) {
        T gr, gi;
        W::unpack(gs[ak], gr, gi);
        br += gf.out(W::mul(gr, gf.re));
        bi += gf.out(W::mul(gi, gf.re));
      }
      wbt[ak] = mk<R>(br, bi);
    }
  }
}

// ---------------------------------------------------------------------------
// JVP for nd <= JVP_CHUNK directions at once, JG of them per pass over the planes
// dwt: [nd][n_omega][M1][N2]; dvt, dut: [nd][n_omega][M][N2]
// ---------------------------------------------------------------------------
template <typename R>
__global__ void __launch_bounds__(DT, 2)
k_diff_jvp(Problem P, DiffTables<R> tab, int nd, const double2* __restrict__ cs,
           const typename Wide<R>::SC* __restrict__ gs, const cx<R>* __restrict__ dwt,
           const double* __restrict__ alpha_arr, const double* __restrict__ dlog_alpha, cx<R>* __restrict__ dvt,
           cx<R>* __restrict__ dut, double* __restrict__ partial) {
  using W = Wide<R>;
  using T = typename W::T;
  __shared__ WC<T> sc[JG][DG][32];
  __shared__ Factor<R> cv_s[JG][32];
  // Phi-dot: the warps' sums (times 2^pexp; joined in FP64 by one thread) and the scalar part
  __shared__ T ps[JG][DG];
  __shared__ int pexp[JG][DG];
  __shared__ double pe[JG];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int om = blockIdx.y, n = P.m1, m = P.m, F = P.n_omega;
  const long long N2 = (long long)P.n * P.n;
  const long long nu = (long long)blockIdx.x * 32 + lane;
  const bool valid = nu < N2;
  const long long at = (long long)om * N2 + (valid ? nu : 0);
  const double ne = tab.ne[at];
  const bool prop = signbit(ne);
  const bool cplx = __any_sync(0xffffffffu, prop);
  const T zero = W::from(0.0);
  WC<T> e[KC], g[KC];
  R big = R(0);
#pragma unroll
  for (int i = 0; i < KC; ++i) {
    const int k = w + DG * i;
    const long long ak = ((long long)om * n + k) * N2 + nu;
    const bool on = valid && k < n;
    e[i] = WC<T>{zero, zero};
    g[i] = WC<T>{zero, zero};
    if (on) {
      e[i].re = W::ld(tab.er + ak);
      if (cplx) e[i].im = W::ld(tab.ei + ak);
      W::unpack(gs[ak], g[i].re, g[i].im);
    }
    big = fmax(big, fmax(fabs(W::r(g[i].re)), fabs(W::r(g[i].im))));
  }
  const int eg = warp_exponent(big);
#pragma unroll
  for (int i = 0; i < KC; ++i) g[i] = WC<T>{scale_by(g[i].re, -eg), scale_by(g[i].im, -eg)};
  ModeScalars s{0.0, 0.0, 1.0};
  double2 c0 = make_double2(0.0, 0.0);
  if (w < JG) {
    s = mode_scalars(tab.tr[at], ne, alpha_arr[om]);
    c0 = cs[at];
  }
#pragma unroll 1
  for (int d0 = 0; d0 < nd; d0 += JG) {
#pragma unroll 1
    for (int jd = 0; jd < JG; ++jd) {
      const int d = d0 + jd;
      if (d >= nd) break;
      cx<R> db[KC];
      R bb = R(0);
#pragma unroll
      for (int i = 0; i < KC; ++i) {
        const int k = w + DG * i;
        db[i] = valid && k < n ? dwt[(((long long)d * F + om) * n + k) * N2 + nu] : czero<R>();
        bb = fmax(bb, fmax(fabs(db[i].x), fabs(db[i].y)));
      }
      const int eb = warp_exponent(bb);
      typename W::Acc cr{}, ci{}, da{};
#pragma unroll
      for (int i = 0; i < KC; ++i) {
        W::mac(cr, e[i].re, db[i].x);
        W::mac(ci, e[i].re, db[i].y);
        if (cplx) {
          W::mac(cr, e[i].im, db[i].y);
          W::mac(ci, W::neg(e[i].im), db[i].x);
        }
        W::mac(da, g[i].re, scale_by(db[i].x, -eb));
        W::mac(da, g[i].im, scale_by(db[i].y, -eb));
      }
      sc[jd][w][lane] = WC<T>{W::sum(cr), W::sum(ci)};
      const T dp = W::wsum(W::sum(da));
      if (lane == 0) {
        ps[jd][w] = dp;
        pexp[jd][w] = eb + eg;
      }
    }
    __syncthreads();
    if (w < JG && d0 + w < nd) {  // warp w: the scalars of direction d0 + w
      const int d = d0 + w;
      T cr = sc[w][0][lane].re, ci = sc[w][0][lane].im;
      for (int i = 1; i < DG; ++i) {
        cr = W::add(cr, sc[w][i][lane].re);
        ci = W::add(ci, sc[w][i][lane].im);
      }
      const double dla = dlog_alpha ? dlog_alpha[d * F + om] : 0.0;
      const double kd = -s.kappa * dla;
      cv_s[w][lane] =
          Factor<R>::make(s.eta * make_double2(W::d(cr) + kd * c0.x, W::d(ci) + kd * c0.y));
      double x = 0.0;
      if (dlog_alpha) x = warp_sum(valid ? 2.0 * s.kappa * s.kappa * s.mu * dla * abs2(c0) : 0.0);
      if (lane == 0) pe[w] = x;
    }
    __syncthreads();
    if (threadIdx.x < JG && d0 + threadIdx.x < nd) {
      double t = pe[threadIdx.x];
      for (int i = 0; i < DG; ++i) t += 2.0 * W::d(ps[threadIdx.x][i]) * pow2d(pexp[threadIdx.x][i]);
      partial[((long long)(d0 + threadIdx.x) * F + om) * gridDim.x + blockIdx.x] = t;
    }
    if (valid) {
      for (int a = w; a < tab.nb; a += DG) {
        const long long ab = ((long long)om * tab.nb + a) * N2 + nu;
        const int jn = min(JG, nd - d0);
        if (!cplx) {
          planes_real<R>(tab, at, ab, a, m, [&](int l, int, T p, T t) {
            const T pt = W::mul(p, t);
#pragma unroll
            for (int jd = 0; jd < JG; ++jd) {
              if (jd < jn) {
                const Factor<R>& cv = cv_s[jd][lane];
                const long long o = (((long long)(d0 + jd) * F + om) * m + l) * N2 + nu;
                dvt[o] = mk<R>(cv.out(W::mulround(p, cv.re)), cv.out(W::mulround(p, cv.im)));
                dut[o] = mk<R>(cv.out(W::mulround(pt, cv.re)), cv.out(W::mulround(pt, cv.im)));
              }
            }
          });
        } else {
          planes_cplx<R>(tab, at, ab, a, m, prop, [&](int l, WC<T> p, WC<T> t) {
#pragma unroll 1
            for (int jd = 0; jd < jn; ++jd) {
              const Factor<R>& cv = cv_s[jd][lane];
              const T vr = W::fma(p.re, cv.re, W::mul(p.im, cv.im));  // conj(P) c
              const T vi = W::fma(p.re, cv.im, W::neg(W::mul(p.im, cv.re)));
              const long long o = (((long long)(d0 + jd) * F + om) * m + l) * N2 + nu;
              dvt[o] = mk<R>(cv.out(vr), cv.out(vi));
              dut[o] = mk<R>(cv.out(W::fma(t.re, vr, W::neg(W::mul(t.im, vi)))),
                             cv.out(W::fma(t.re, vi, W::mul(t.im, vr))));
            }
          });
        }
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// step 3 and its derivatives, one thread per voxel (X planes), arrays
// [n_omega][M N^2] (fields) and [M N^2] (xi)
// ---------------------------------------------------------------------------
template <typename R>
__global__ void k_diff_combine(Problem P, const cx<R>* __restrict__ Vx, const cx<R>* __restrict__ ux,
                               R* __restrict__ xi, R* __restrict__ c, R* __restrict__ xis) {
  const long long MN2 = (long long)P.m * P.n * P.n;
  const R guard2 = (R)(P.eps_u * P.eps_u * P.n_omega);
  const R ic2 = (R)(1.0 / (P.c0 * P.c0));
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < MN2; p += (long long)gridDim.x * blockDim.x) {
    R num = 0, D = 0;
    for (int om = 0; om < P.n_omega; ++om) {
      const cx<R> u = ux[om * MN2 + p], V = Vx[om * MN2 + p];
      num += u.x * V.x + u.y * V.y;
      D += u.x * u.x + u.y * u.y;
    }
    const R x = D < guard2 ? R(0) : num / D;
    xi[p] = x;
    xis[p] = x;
    if (c) c[p] = x < ic2 ? R(1) / sqrt(ic2 - x) : R(NAN);
  }
}

template <typename R>
__global__ void k_diff_vjp_point(Problem P, const R* __restrict__ gxi, const cx<R>* __restrict__ Vx,
                                 const cx<R>* __restrict__ ux, const R* __restrict__ xis, cx<R>* __restrict__ Vb,
                                 cx<R>* __restrict__ ub) {
  const long long MN2 = (long long)P.m * P.n * P.n;
  const R guard2 = (R)(P.eps_u * P.eps_u * P.n_omega);
  for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < MN2; p += (long long)gridDim.x * blockDim.x) {
    R D = 0;
    for (int om = 0; om < P.n_omega; ++om) D += abs2(ux[om * MN2 + p]);
    const R gx = D < guard2 ? R(0) : gxi[p] / D;
    const R x2 = R(2) * xis[p];
    for (int om = 0; om < P.n_omega; ++om) {
      const cx<R> u = ux[om * MN2 + p], V = Vx[om * MN2 + p];
      Vb[om * MN2 + p] = gx * u;
      ub[om * MN2 + p] = gx * (V - x2 * u);
    }
  }
}

// out[r] = sum_c partial[r cols + c]: one warp per row, lanes over the columns, then a
// tree over the lanes (a fixed order)
__global__ void k_reduce_rows(const double* __restrict__ partial, int rows, int cols, double* __restrict__ out) {
  const int r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (r >= rows) return;
  double s = 0.0;
  for (int c = lane; c < cols; c += 32) s += partial[(long long)r * cols + c];
  s = warp_sum(s);
  if (lane == 0) out[r] = s;
}

unsigned point_grid(long long n) {
  const long long b = (n + 255) / 256;
  const long long cap = 8LL * sm_count();
  return (unsigned)(b < cap ? (b > 0 ? b : 1) : cap);
}

}  // namespace

int diff_blocks_per_omega(int n) { return (int)(((long long)n * n + 31) / 32); }

template <typename R>
size_t diff_tables(const Problem& P, void* base, DiffTables<R>* tab, DiffTablesOut<R>* out) {
  using S = typename DiffTables<R>::S;
  const size_t F = P.n_omega, N2 = (size_t)P.n * P.n, nb = (P.m + DIFF_PB - 1) / DIFF_PB;
  char* b = (char*)base;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* p = b + off;
    off = (off + bytes + 255) & ~(size_t)255;
    return p;
  };
  DiffTablesOut<R> o;
  o.er = (S*)take(sizeof(S) * F * P.m1 * N2);
  o.ei = (S*)take(sizeof(S) * F * P.m1 * N2);
  o.pr = (S*)take(sizeof(S) * F * nb * N2);
  o.pi = (S*)take(sizeof(S) * F * nb * N2);
  o.sr = (S*)take(sizeof(S) * F * nb * N2);
  o.si = (S*)take(sizeof(S) * F * nb * N2);
  o.q = (typename DiffTables<R>::S2*)take(2 * sizeof(S) * F * N2);
  o.g = (S*)take(sizeof(S) * F * N2);
  o.tr = (double*)take(8 * F * N2);
  o.ne = (double*)take(8 * F * N2);
  o.inc = (double2*)take(16 * F * P.m);
  if (out) *out = o;
  if (tab) *tab = DiffTables<R>{o.er, o.ei, o.pr, o.pi, o.sr, o.si, o.q, o.g, o.tr, o.ne, o.inc, (int)nb};
  return off;
}

template <typename R>
cudaError_t launch_diff_tables(const Problem& P, const DiffTables<R>& tab, const DiffTablesOut<R>& out,
                               cudaStream_t s) {
  k_diff_tables<R><<<dim3(diff_blocks_per_omega(P.n), P.n_omega), DT, 0, s>>>(P, tab, out);
  k_diff_incident<<<P.n_omega, 64, 0, s>>>(P, out.inc);
  return cudaGetLastError();
}

cudaError_t launch_diff_alpha(const double* log_alpha, int F, double* la, cudaStream_t s) {
  k_diff_alpha<<<1, MAX_OMEGA, 0, s>>>(log_alpha, F, la);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_diff_forward(const Problem& P, const DiffTables<R>& tab, const cx<R>* wt, const double* alpha,
                                double2* cs, void* gs, cx<R>* vt, cx<R>* ut, double* partial,
                                unsigned long long* ctr, cudaStream_t s) {
  k_diff_forward<R><<<dim3(diff_blocks_per_omega(P.n), P.n_omega), DT, 0, s>>>(
      P, tab, wt, alpha, cs, (typename Wide<R>::SC*)gs, vt, ut, partial, ctr);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_diff_vjp(const Problem& P, const DiffTables<R>& tab, const double2* cs, const void* gs,
                            const cx<R>* vbt, const cx<R>* ubt, const double* alpha, const double* grad_phi,
                            cx<R>* wbt, double* partial, cudaStream_t s) {
  k_diff_vjp<R><<<dim3(diff_blocks_per_omega(P.n), P.n_omega), DT, 0, s>>>(
      P, tab, cs, (const typename Wide<R>::SC*)gs, vbt, ubt, alpha, grad_phi, wbt, partial);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_diff_jvp(const Problem& P, const DiffTables<R>& tab, int nd, const double2* cs, const void* gs,
                            const cx<R>* dwt, const double* alpha, const double* dlog_alpha, cx<R>* dvt, cx<R>* dut,
                            double* partial, cudaStream_t s) {
  if (nd < 1 || nd > JVP_CHUNK) return cudaErrorInvalidValue;
  k_diff_jvp<R><<<dim3(diff_blocks_per_omega(P.n), P.n_omega), DT, 0, s>>>(
      P, tab, nd, cs, (const typename Wide<R>::SC*)gs, dwt, alpha, dlog_alpha, dvt, dut, partial);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_diff_combine(const Problem& P, const cx<R>* Vx, const cx<R>* ux, R* xi, R* c, R* xis,
                                cudaStream_t s) {
  k_diff_combine<R><<<point_grid((long long)P.m * P.n * P.n), 256, 0, s>>>(P, Vx, ux, xi, c, xis);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_diff_vjp_point(const Problem& P, const R* gxi, const cx<R>* Vx, const cx<R>* ux, const R* xis,
                                  cx<R>* Vb, cx<R>* ub, cudaStream_t s) {
  k_diff_vjp_point<R><<<point_grid((long long)P.m * P.n * P.n), 256, 0, s>>>(P, gxi, Vx, ux, xis, Vb, ub);
  return cudaGetLastError();
}

cudaError_t launch_reduce_rows(const double* partial, int rows, int cols, double* out, cudaStream_t s) {
  k_reduce_rows<<<(rows + 3) / 4, 128, 0, s>>>(partial, rows, cols, out);
  return cudaGetLastError();
}

#define FL_DIFF_INST(R)                                                                                            \
  template size_t diff_tables<R>(const Problem&, void*, DiffTables<R>*, DiffTablesOut<R>*);                         \
  template cudaError_t launch_diff_tables<R>(const Problem&, const DiffTables<R>&, const DiffTablesOut<R>&,         \
                                             cudaStream_t);                                                        \
  template cudaError_t launch_diff_forward<R>(const Problem&, const DiffTables<R>&, const cx<R>*, const double*,    \
                                              double2*, void*, cx<R>*, cx<R>*, double*, unsigned long long*,       \
                                              cudaStream_t);                                                       \
  template cudaError_t launch_diff_vjp<R>(const Problem&, const DiffTables<R>&, const double2*, const void*,        \
                                          const cx<R>*, const cx<R>*, const double*, const double*, cx<R>*,        \
                                          double*, cudaStream_t);                                                  \
  template cudaError_t launch_diff_jvp<R>(const Problem&, const DiffTables<R>&, int, const double2*, const void*,   \
                                          const cx<R>*, const double*, const double*, cx<R>*, cx<R>*, double*,     \
                                          cudaStream_t);                                                           \
  template cudaError_t launch_diff_combine<R>(const Problem&, const cx<R>*, const cx<R>*, R*, R*, R*,               \
                                              cudaStream_t);                                                       \
  template cudaError_t launch_diff_vjp_point<R>(const Problem&, const R*, const cx<R>*, const cx<R>*, const R*,     \
                                                cx<R>*, cx<R>*, cudaStream_t);
FL_DIFF_INST(double)
FL_DIFF_INST(float)
#undef FL_DIFF_INST

}  // namespace fl
