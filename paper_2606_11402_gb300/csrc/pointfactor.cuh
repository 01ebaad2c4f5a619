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
// Group form: a group of G lanes of one warp (G = 8, 16 or 32 >= k), lane a
// holding row a of M in registers.  Left-looking Cholesky: at step j every
// lane forms its Schur value t_a = M_aj - sum_{m<j} L_am L_jm from its own
// row and row j of L (published in shared memory by lane j at earlier
// steps); lane j's t is the pivot.  The forward solve y = L^-1 m rides along,
// sigma^2 = Var(w) - y.y accumulates in compensated FP32 (exact two-product,
// two-sum), and beta = L^-T y is a backward sweep over L's columns.  Rows and
// columns k..G-1 are identity padding.  Shared by the factor kernel and the
// adjoint kernels, which recompute the factors instead of storing them, so
// that both see bit-identical b and sigma.
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

template <int G>
struct PointState {
  float A[G];      // row a of M, then of L (lower part valid)
  float D2[G];     // squared distances |x_a - x_b|^2 of row a
  float d2q;       // |x_a - x_i|^2
  float inv_own;   // 1 / L_aa
  float y_own;     // y_a
  float b_own;     // b_a (covariance-form weight of neighbour a)
  float sigma;     // conditional standard deviation (same on all lanes)
  bool clamped;    // a pivot was floored (same on all lanes)
  float max_ratio; // max_j M_jj / pivot_j (same on all lanes)
  float varw;      // Var(w) (same on all lanes)
  bool inc;        // increment form (same on all lanes)
};

// Shared-memory row stride and per-group footprint (floats) for G lanes.
template <int G>
struct PFLayout {
  static constexpr int SG = G + 4;
  static constexpr int GS = G * SG + 4;
};

template <int G, int KT>
__device__ __forceinline__ void point_factor_group(PointState<G>& st, int a, int k,
                                                   const KernF& kf, float4 xa, float4 xq,
                                                   float* Lg) {
  constexpr int SG = PFLayout<G>::SG;
  const unsigned full = 0xffffffffu;
  const bool real = a < k;
  const float k0 = kf.s2 + kf.nug;
  const float nug = kf.nug;
  st.d2q = sqdist(xa, xq);
  const KG qa = kappa_gamma_d2<KT>(kf, st.d2q);
  st.inc = __shfl_sync(full, qa.g, 0, G) < 0.5f * kf.s2;
  const bool inc = st.inc;
  const float eai = inc ? qa.g : qa.k;  // entry (a, i) before the change of variables
  const float e0i = __shfl_sync(full, eai, 0, G);
  float ea0 = 0.0f;  // entry (a, 0)
#pragma unroll
  for (int bcol = 0; bcol < G; bcol++) {
    float bx = __shfl_sync(full, xa.x, bcol, G);
    float by = __shfl_sync(full, xa.y, bcol, G);
    float bz = __shfl_sync(full, xa.z, bcol, G);
    float dx = xa.x - bx, dy = xa.y - by, dz = xa.z - bz;
    float d2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
    st.D2[bcol] = d2;
    const KG kg = kappa_gamma_d2<KT>(kf, d2);
    const float ev = inc ? kg.g : kg.k;
    if (bcol == 0) ea0 = ev;
    const float e0b = __shfl_sync(full, ev, 0, G);  // entry (0, bcol) from row 0
    const bool both = real && bcol < k;
    float m;
    if (bcol == a) {
      m = real ? ((a == 0 || !inc) ? k0 : 2.0f * (ea0 + nug)) : 1.0f;
    } else if (!inc) {
      m = ev;
    } else if (a == 0) {
      m = -(e0b + nug);
    } else if (bcol == 0) {
      m = -(ea0 + nug);
    } else {
      m = ((ea0 + e0b) - ev) + nug;
    }
    st.A[bcol] = both || bcol == a ? m : 0.0f;
  }
  float c = !real ? 0.0f
                  : !inc ? eai : (a == 0 ? -(e0i + nug) : ((ea0 + e0i) - eai) + nug);
  st.varw = inc ? 2.0f * (e0i + nug) : k0;
  DF s2{st.varw, 0.0f};
  const float pfloor = kPdFloor * k0;
  st.clamped = false;
  st.max_ratio = 1.0f;
  st.inv_own = 1.0f;
  st.y_own = 0.0f;
#pragma unroll
  for (int j = 0; j < G; j++) {
    if (j >= k) break;
    float tv = st.A[j];
    float t2 = 0.0f;
#pragma unroll
    for (int m = 0; m + 4 <= j; m += 4) {
      float4 r = *reinterpret_cast<const float4*>(Lg + j * SG + m);
      tv = fmaf(-st.A[m], r.x, tv);
      t2 = fmaf(-st.A[m + 1], r.y, t2);
      tv = fmaf(-st.A[m + 2], r.z, tv);
      t2 = fmaf(-st.A[m + 3], r.w, t2);
    }
#pragma unroll
    for (int m = (j / 4) * 4; m < j; m++) tv = fmaf(-st.A[m], Lg[j * SG + m], tv);
    const float mjj = __shfl_sync(full, st.A[j], j, G);
    tv += t2;
    float piv = __shfl_sync(full, tv, j, G);
    if (!(piv > pfloor)) {
      piv = pfloor;
      st.clamped = true;
    }
    float ljj = sqrt_newton(piv);
    float inv = rcp_newton(ljj);
    st.max_ratio = fmaxf(st.max_ratio, mjj * inv * inv);
    float laj = (a == j) ? ljj : tv * inv;
    st.A[j] = laj;
    if (a == j) st.inv_own = inv;
    Lg[a * SG + j] = laj;
    float yj = __shfl_sync(full, c, j, G) * inv;
    if (a == j) st.y_own = yj;
    if (a > j) c = fmaf(-laj, yj, c);
    s2 = df_sub_square(s2, yj);
    __syncwarp(full);
  }
  float sig2 = s2.hi + s2.lo;
  if (!(sig2 > pfloor)) {
    sig2 = pfloor;
    st.clamped = true;
  }
  st.sigma = sqrtf(sig2);
  // beta = L^-T y, last entry first; lane a keeps d_a = y_a - sum_{m>a} L_ma beta_m
  float d = st.y_own;
  st.b_own = 0.0f;
#pragma unroll
  for (int j = G - 1; j >= 0; j--) {
    if (j >= k) continue;
    float bj = __shfl_sync(full, d * st.inv_own, j, G);
    if (a == j) st.b_own = bj;
    if (a < j) d = fmaf(-Lg[j * SG + a], bj, d);
  }
  // increment form: b_0 = 1 + beta_0 - sum_{a>=1} beta_a (summed in lane order)
  float sb = 0.0f;
#pragma unroll
  for (int j = 1; j < G; j++) sb += __shfl_sync(full, st.b_own, j, G);
  if (a == 0 && inc) st.b_own = (1.0f + st.b_own) - sb;
}

// Solves K_cc g = r for the factor held by the group (L rows in st.A and in
// Lg): g = T^T M^-1 T r.  Lane a supplies r_a (zero for a >= k) and receives
// g_a.
template <int G>
__device__ __forceinline__ float group_chol_solve(const PointState<G>& st, int a, int k,
                                                  float r, const float* Lg) {
  constexpr int SG = PFLayout<G>::SG;
  const unsigned full = 0xffffffffu;
  const float r0 = __shfl_sync(full, r, 0, G);
  if (st.inc && a >= 1 && a < k) r -= r0;
  float z_own = 0.0f;
#pragma unroll
  for (int j = 0; j < G; j++) {
    if (j >= k) break;
    float zj = __shfl_sync(full, r * st.inv_own, j, G);
    if (a == j) z_own = zj;
    if (a > j) r = fmaf(-st.A[j], zj, r);
  }
  float d = z_own, g_own = 0.0f;
#pragma unroll
  for (int j = G - 1; j >= 0; j--) {
    if (j >= k) continue;
    float gj = __shfl_sync(full, d * st.inv_own, j, G);
    if (a == j) g_own = gj;
    if (a < j) d = fmaf(-Lg[j * SG + a], gj, d);
  }
  float sg = 0.0f;
#pragma unroll
  for (int j = 1; j < G; j++) sg += __shfl_sync(full, g_own, j, G);
  if (a == 0 && st.inc) g_own -= sg;
  return g_own;
}

template <int I, int N, class F>
__device__ __forceinline__ void static_for(F&& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    static_for<I + 1, N>(f);
  }
}

}  // namespace ggp
