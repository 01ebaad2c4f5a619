// Per-point conditional factor of Sec. 2.1 Eq. 2 in FP32: the weights
// b_i = K_ic K_cc^-1 and sigma_i^2 = K_ii - K_ic K_cc^-1 K_ci.
//
// Increment form.  Where neighbours are close on the scale of the
// lengthscale, every entry of K_cc is close to kappa(0): FP32 keeps only the
// leading digits of kappa(r), and the Cholesky of K_cc then cancels them
// (condition numbers of 1e5-1e11 on the measured clouds).  Such rows are
// factored in increments of the field instead, an exact change of variables:
// with c_0 the nearest neighbour, z_0 = x(c_0), z_a = x(c_a) - x(c_0)
// (a >= 1) and the target w = x(i) - x(c_0),
//   M_00 = kappa(0) + nugget,       M_a0 = -(g_a0 + nugget),
//   M_ab = (g_a0 + g_b0) - g_ab + nugget (1 + [a = b]),
//   m_0  = -(g_0i + nugget),        m_a  = (g_a0 + g_0i) - g_ai + nugget,
//   Var(w) = 2 (g_0i + nugget),
// where g = kappa(0) - kappa(r) is the variogram, evaluated with a small
// relative error even as r -> 0 (gamma_d2).  With L = chol(M),
// y = L^-1 m and beta = L^-T y, E[w | z] = beta . z gives the weights
// b_a = beta_a (a >= 1), b_0 = 1 + beta_0 - sum_{a>=1} beta_a, and
// sigma^2 = Var(w) - y.y.  The change of variables is unit lower triangular,
// so the pivots of M equal those of K_cc (conditional variances) and the
// floor policy below is the covariance form's; only the rounding differs.
// K_cc^-1 r (the backward) is T^T M^-1 T r with (T r)_a = r_a - r_0.
// A row whose nearest neighbour is far (g_0i >= kappa(0) / 2) has small
// weights, which the recovery of b_0 would swamp with its rounding error; it
// keeps the covariance form (M = K_cc, m = K_ci, Var(w) = K_ii, b = beta,
// T = identity).  The choice is made per row from g_0i.
//
// A pivot at or below 1e-7 of kappa(0) + nugget is raised to that floor and
// flagged; so is sigma^2.  max_ratio = max_j M_jj / pivot_j (pivot after the
// floor) bounds the scaled condition number of M from below and gives the
// row's error estimate (rescue.cuh).
//
// The factor is a left-looking Cholesky with two accumulators per entry (m =
// 0, 2 and m = 1, 3 mod 4 over whole blocks of four, the rest on the first):
// t_aj = M_aj - sum_{m<j} L_am L_jm, L_aj = t_aj / L_jj; the forward solve y =
// L^-1 m rides along, sigma^2 = Var(w) - y.y accumulates in compensated FP32
// (exact two-product, two-sum), and beta = L^-T y is a backward sweep.  Rows
// and columns past k are identity padding.  Two lanes per point for k <= 16
// (pointpair.cuh), eight for k <= 32 (pointoct.cuh), a warp with the matrix in
// shared memory above (pointwide.cuh); the adjoint and on-the-fly kernels
// recompute the factors with the same code, so that all see the same bits.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "rescue.cuh"

namespace ggp {

constexpr float kPdFloor = 1e-7f;

// Running product of sigma^2 values in FP64 with a separate binary exponent
// (one log per thread at the end).
struct LogAcc {
  double m = 1.0;
  int e = 0;
  __device__ void mul(float sigma) {
    m *= (double)sigma * (double)sigma;
    int ex;
    m = frexp(m, &ex);
    e += ex;
  }
  __device__ double log_value() const { return log(m) + (double)e * 0.69314718055994530942; }
};

// Block-wide FP64 sum (blockDim.x a multiple of 32, at most 1024), added to
// *out.  The trailing barrier lets a kernel call it again at once: the
// shared partials are not overwritten while thread 0 still reads them.
__device__ inline void block_add_double(double v, double* out) {
  __shared__ double red[32];
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); i++) s += red[i];
    atomicAdd(out, s);
  }
  __syncthreads();
}

struct DF {  // double-float: value = hi + lo
  float hi, lo;
};

__device__ __forceinline__ DF df_sub_square(DF s, float y) {
  float p = __fmul_rn(y, y);
  float e = __fmaf_rn(y, y, -p);  // p + e == y*y exactly
  float t = __fsub_rn(s.hi, p);
  float bb = __fsub_rn(t, s.hi);
  float err = __fadd_rn(__fsub_rn(s.hi, __fsub_rn(t, bb)), __fsub_rn(-p, bb));
  float lo = __fsub_rn(__fadd_rn(s.lo, err), e);
  float h = __fadd_rn(t, lo);
  float l = __fsub_rn(lo, __fsub_rn(h, t));
  return DF{h, l};
}

template <int I, int N, class F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    static_for<I + 1, N>(f);
  }
}

}  // namespace ggp
