// Internal interface of the fixed-alpha derivative kernels (diff.cu) used by the
// C-ABI layer; the public interface is include/flatlayer_diff.h.
#pragma once

#include "pipeline.cuh"

namespace fl {

constexpr int JVP_CHUNK = 16;  // directions per JVP launch
constexpr int DIFF_PB = 8;     // X planes between two tabulated values of P and T

// The geometry of every mode (diff.cu), [n_omega][..][N^2] with the mode fastest: e
// [M1], the values of P and gamma times the sums of T at one plane of each block of DIFF_PB
// planes [nb], q, |gamma| with its sign, tr, ||E|| (negative: propagating) and the incident
// plane wave's U~0 at nu = 0 [M].  One component is a double, or two floats (high part,
// remainder) in the mixed precision.
template <typename R> struct DiffStore;
template <> struct DiffStore<double> { using S = double; };
template <> struct DiffStore<float> { using S = float2; };
template <typename R> struct DiffTables {
  using S = typename DiffStore<R>::S;
  struct S2 { S x, y; };
  const S *er, *ei, *pr, *pi, *sr, *si;
  const S2* q;
  const S* g;
  const double *tr, *ne;
  const double2* inc;
  int nb;
};
template <typename R> struct DiffTablesOut {
  using S = typename DiffStore<R>::S;
  S *er, *ei, *pr, *pi, *sr, *si;
  typename DiffTables<R>::S2* q;
  S* g;
  double *tr, *ne;
  double2* inc;
};
// carves the tables at `base` (null: only counts); returns their bytes
template <typename R>
size_t diff_tables(const Problem& P, void* base, DiffTables<R>* tab, DiffTablesOut<R>* out);

// blocks per frequency of the per-mode kernels (fixed for a shape, so that the per-block
// partial sums, and hence the results, are reproducible)
int diff_blocks_per_omega(int n);

template <typename R>
cudaError_t launch_diff_tables(const Problem& P, const DiffTables<R>& tab, const DiffTablesOut<R>& out,
                               cudaStream_t s);
// la[0..F) <- log alpha, la[F..2F) <- alpha
cudaError_t launch_diff_alpha(const double* log_alpha, int F, double* la, cudaStream_t s);
template <typename R>
cudaError_t launch_diff_forward(const Problem& P, const DiffTables<R>& tab, const cx<R>* wt, const double* alpha,
                                double2* cs, void* gs, cx<R>* vt, cx<R>* ut, double* partial,
                                unsigned long long* ctr, cudaStream_t s);
template <typename R>
cudaError_t launch_diff_vjp(const Problem& P, const DiffTables<R>& tab, const double2* cs, const void* gs,
                            const cx<R>* vbt, const cx<R>* ubt, const double* alpha, const double* grad_phi,
                            cx<R>* wbt, double* partial, cudaStream_t s);
template <typename R>
cudaError_t launch_diff_jvp(const Problem& P, const DiffTables<R>& tab, int nd, const double2* cs, const void* gs,
                            const cx<R>* dwt, const double* alpha, const double* dlog_alpha, cx<R>* dvt, cx<R>* dut,
                            double* partial, cudaStream_t s);
template <typename R>
cudaError_t launch_diff_combine(const Problem& P, const cx<R>* Vx, const cx<R>* ux, R* xi, R* c, R* xis,
                                cudaStream_t s);
template <typename R>
cudaError_t launch_diff_vjp_point(const Problem& P, const R* gxi, const cx<R>* Vx, const cx<R>* ux, const R* xis,
                                  cx<R>* Vb, cx<R>* ub, cudaStream_t s);
// dxi of step 3 for nd directions: the inverse transform along x of dV~, dU~ ([nd][n_omega][M][N][N],
// already transformed along y) with the pointwise derivative (fft_forward.cu)
template <typename R>
cudaError_t launch_diff_jvp_rows(const Problem& P, int nd, const cx<R>* dv, const cx<R>* du, const cx<R>* Vx,
                                 const cx<R>* ux, const R* xis, R* dxi, const cx<R>* tw, cudaStream_t s);
cudaError_t launch_reduce_rows(const double* partial, int rows, int cols, double* out, cudaStream_t s);

}  // namespace fl
