// Per-point conditional factor for k <= 16: two lanes per point.
//
// The arithmetic is that of pointfactor.cuh (increment or covariance form,
// left-looking Cholesky with two accumulators, forward solve riding along,
// compensated sigma^2, backward sweep), element by element and in the order
// given there.  (In the covariance form the registers hold -kappa, so a value
// that underflows is a zero of the other sign.)  Lane r of a point's pair owns the rows a = 2 s + r (slot s) of M, as packed pairs of
// columns in registers; row j of L goes to shared memory when it is complete
// and both lanes read it back for step j and for the backward sweep.
//
// What bounds these kernels is instruction issue: a k = 16 row takes 152
// covariance values, each a square root, an exponential and a polynomial.
// Three choices follow.
//  * Every covariance value, product and update is a packed FP32 pair
//    (fma.rn.f32x2 and its kin: two roundings, one instruction), and no step
//    of a value branches: gamma's polynomial and closed forms are both
//    evaluated and selected, and a row in the covariance form runs through the
//    same instructions with other constants.
//  * The registers hold -M and the updates add L L^T to it, so no operand is
//    ever negated.
//  * Two lanes per point need 36 register pairs for the matrix instead of one
//    thread's 136 registers, and the matrix is built in registers: 850 bytes
//    of shared memory per point.  An SM holds 12 warps (16 for K <= 12)
//    instead of the 8 of one thread per point, where each scheduler had 2
//    warps to choose from.
// Measured (K = 16, Matern-3/2, unit-Gaussian points): the factor of 2^20 rows
// takes 13,000 -> 8,100 warp instructions per 32 rows; 2^24 rows, with the
// dense block and the export, 16.2 -> 9.4 ms; one fit step (value and
// gradient in one pass) at 2^22 7.9 -> 4.9 ms.  A packed operation takes two
// issue cycles on this part, so the packing itself saves decoding and code
// size, not issue slots.
#pragma once

#include "pointfactor.cuh"
#include "sweepsync.cuh"

namespace ggp {

__device__ __forceinline__ float2 two(float x) { return make_float2(x, x); }

// Constants of a row's covariance values.  value = s2 (a < sw ? near : far):
// gamma in the increment form; in the covariance form near is never taken and
// far = 0 - kappa / s2, so the value is -kappa.
struct RowForm {
  float sw, one;
};

// sqrt_newton of two arguments.
__device__ __forceinline__ float2 sqrt_pair(float2 d2) {
  float2 y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(d2.x));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(d2.y));
  y.x = fminf(y.x, 9.2233720e18f);
  y.y = fminf(y.y, 9.2233720e18f);
  const float2 g = __fmul2_rn(d2, y), h = __fmul2_rn(two(0.5f), y);
  return __ffma2_rn(__ffma2_rn(make_float2(-g.x, -g.y), g, d2), h, g);
}

// cov_arg of two squared distances.
template <int KT>
__device__ __forceinline__ float2 arg_pair(const KernF& kf, float2 d2) {
  if (KT == GRAPHGP_SQEXP)
    return __fmul2_rn(__fmul2_rn(__fmul2_rn(two(0.5f), d2), two(kf.inv_ell)), two(kf.inv_ell));
  float2 a = sqrt_pair(d2);
  if (KT == GRAPHGP_MATERN32) a = __fmul2_rn(two(1.7320508075688772f), a);
  if (KT == GRAPHGP_MATERN52) a = __fmul2_rn(two(2.2360679774997896f), a);
  return __fmul2_rn(a, two(kf.inv_ell));
}

// Two covariance values from two squared distances: the values of gamma_at
// (increment form) or -kappa_at (covariance form) in packed arithmetic.
template <int KT>
__device__ __forceinline__ float2 entry_pair(const KernF& kf, RowForm rf, float2 d2) {
  const float2 a = arg_pair<KT>(kf, d2);
  const float2 e = make_float2(expf(-a.x), expf(-a.y));
  float2 near, far;
  if (KT == GRAPHGP_SQEXP || KT == GRAPHGP_MATERN12) {
    near = __fmul2_rn(a, poly_exp1_2(a));
    far = __ffma2_rn(e, two(-1.0f), two(rf.one));
  } else {
    const float2 aa = __fmul2_rn(a, a);
    float2 p = __fadd2_rn(two(1.0f), a);
    if (KT == GRAPHGP_MATERN32) {
      near = __fmul2_rn(__fmul2_rn(aa, poly_m32_2(a)), e);
    } else {
      near = __fmul2_rn(__fmul2_rn(aa, poly_m52_2(a)), e);
      p = __ffma2_rn(aa, two(1.0f / 3.0f), p);
    }
    far = __ffma2_rn(__fmul2_rn(p, e), two(-1.0f), two(rf.one));
  }
  return __fmul2_rn(two(kf.s2), make_float2(a.x < rf.sw ? near.x : far.x,
                                            a.y < rf.sw ? near.y : far.y));
}

// Shared memory of one point: x[K], y[K], z[K] of its neighbours, then the
// rows of L, row a at row_off(a) with a + 1 entries (the diagonal one holds
// 1 / L_aa) padded to 16 bytes.  The stride is an odd multiple of four
// floats, so the 16-byte reads of a warp's points fall on different banks.
constexpr int kPairThreads = 128;

template <int K>
struct PairLayout {
  static constexpr int R = K / 2;  // rows per lane
  static __host__ __device__ constexpr int row_off(int a) {
    return 3 * K + 8 * (a / 4) * (a / 4 + 1) + 4 * (a % 4) * (a / 4 + 1);
  }
  static constexpr int kUsed = row_off(K);
  static constexpr int kStride = kUsed / 4 % 2 ? kUsed : kUsed + 4;
  static constexpr int kPoints = kPairThreads / 2;  // points per block
  static constexpr size_t kBytes = (size_t)kPoints * kStride * sizeof(float);
  // Blocks per SM that the registers allow: 128 per thread spill at K = 16
  // (2^23 rows: 3.9 ms with four blocks, 3.5 ms with three)
  static constexpr int kBlocks = K > 12 ? 3 : 4;
};

// Persistent grid: every block resident.
template <int K>
inline unsigned pair_grid(int64_t npts) {
  const int64_t blocks = (npts + PairLayout<K>::kPoints - 1) / PairLayout<K>::kPoints;
  const int64_t most = (int64_t)PairLayout<K>::kBlocks * num_sms();
  return (unsigned)(blocks < most ? blocks : most);
}

// State of a point's factor: the lane's rows of L and, on both lanes alike,
// the weights and the conditional standard deviation.
template <int K>
struct PairFactor {
  static constexpr int R = K / 2;
  float2 A[R * (R + 1) / 2];  // slot s, columns 2c, 2c + 1 at ap(s, c)
  float2 b[K / 2];            // y = L^-1 m, beta = L^-T y, then b (zero past k)
  float sigma, max_ratio, varw;
  bool clamped, inc, finite;
  static __host__ __device__ constexpr int ap(int s, int c) { return s * (s + 1) / 2 + c; }
  __device__ __forceinline__ float weight(int a) const { return a & 1 ? b[a / 2].y : b[a / 2].x; }
};

// The neighbour coordinates of a row on their way to shared memory: K / 2 per
// lane, in chunks of four (padding entries are index 0).
template <int K>
struct PairLoad {
  static constexpr int Q = (K + 4) / 8;
  int4 n[Q];
  float4 x[4 * Q];
  __device__ __forceinline__ void indices(int r, const int32_t* __restrict__ row) {
#pragma unroll
    for (int q = 0; q < Q; q++)
      if (4 * (2 * q + r) < K) n[q] = __ldg(reinterpret_cast<const int4*>(row) + 2 * q + r);
  }
  __device__ __forceinline__ void coords(int r, const float4* __restrict__ xs) {
#pragma unroll
    for (int q = 0; q < Q; q++)
      if (4 * (2 * q + r) < K) {
        x[4 * q] = __ldg(xs + n[q].x);
        x[4 * q + 1] = __ldg(xs + n[q].y);
        x[4 * q + 2] = __ldg(xs + n[q].z);
        x[4 * q + 3] = __ldg(xs + n[q].w);
      }
  }
  // between warp barriers: earlier readers of S are done, later ones wait
  __device__ __forceinline__ void stage(float* S, int r) const {
    __syncwarp();
#pragma unroll
    for (int q = 0; q < Q; q++) {
      const int c = 2 * q + r;
      if (4 * c < K) {
        const float4* u = x + 4 * q;
        *reinterpret_cast<float4*>(S + 4 * c) = make_float4(u[0].x, u[1].x, u[2].x, u[3].x);
        *reinterpret_cast<float4*>(S + K + 4 * c) = make_float4(u[0].y, u[1].y, u[2].y, u[3].y);
        *reinterpret_cast<float4*>(S + 2 * K + 4 * c) = make_float4(u[0].z, u[1].z, u[2].z, u[3].z);
      }
    }
    __syncwarp();
  }
};

__device__ __forceinline__ float2 sqdist2(float2 dx, float2 dy, float2 dz) {
  return __ffma2_rn(dz, dz, __ffma2_rn(dy, dy, __fmul2_rn(dx, dx)));
}

__device__ __forceinline__ float2 sub2(float x, float2 y) {
  return __ffma2_rn(y, two(-1.0f), two(x));  // exact product: one rounding
}

// y <- L^-T y with the rows of L in shared memory, last entry first, the whole
// vector on both lanes.
template <int K>
__device__ __forceinline__ void pair_back_solve(const float* S, float2 (&y)[K / 2]) {
  static_for<0, K>([&](auto Jr) {
    constexpr int j = K - 1 - decltype(Jr)::value;
    float2 Lj[(j + 4) / 4 * 2];
#pragma unroll
    for (int c = 0; c < (j + 4) / 4; c++) {
      const float4 q =
          *reinterpret_cast<const float4*>(S + PairLayout<K>::row_off(j) + 4 * c);
      Lj[2 * c] = make_float2(q.x, q.y);
      Lj[2 * c + 1] = make_float2(q.z, q.w);
    }
    const float bj = j & 1 ? y[j / 2].y * Lj[j / 2].y : y[j / 2].x * Lj[j / 2].x;
    if (j & 1) y[j / 2].y = bj; else y[j / 2].x = bj;
#pragma unroll
    for (int c = 0; c < j / 2; c++) y[c] = __ffma2_rn(Lj[c], two(-bj), y[c]);
    if (j & 1) y[j / 2].x = __fmaf_rn(Lj[j / 2].x, -bj, y[j / 2].x);
  });
}

// `late` runs when the last rows of L are being formed and `done` when L is
// complete: the caller starts the loads of its next point there (the
// registers of the finished rows are free).
struct NoHook {
  __device__ __forceinline__ void operator()() const {}
};

template <int K, int KT, class Late = NoHook, class Done = NoHook>
__device__ __forceinline__ void pair_factor(PairFactor<K>& f, float* S, int r, int k,
                                            const KernF& kf, float4 xq, Late late = Late(),
                                            Done done = Done()) {
  using PL = PairLayout<K>;
  using PF = PairFactor<K>;
  constexpr int R = K / 2;
  const unsigned full = 0xffffffffu;
  const float k0 = kf.s2 + kf.nug, nug = kf.nug;
  const float g0i = gamma_at<KT>(
      kf, cov_arg<KT>(kf, sqdist(make_float4(S[0], S[K], S[2 * K], 0.0f), xq)));
  const bool inc = g0i < 0.5f * kf.s2;
  f.inc = inc;
  const RowForm rf{inc ? cov_switch<KT>() : -1.0f, inc ? 1.0f : 0.0f};
  // Covariance values, left in the rows' place by rolled loops (unrolled, the
  // code exceeds the instruction cache).  Blocks of four rows by four columns
  // left of the diagonal, two rows per lane; then the diagonal blocks and the
  // values with the point (put in the rows' diagonal place), two blocks per
  // step: of a block's six pairs lane 0 takes column 0, lane 1 the others.
#pragma unroll 1
  for (int t = 1; 4 * t < k; t++) {
    const float* Xa = S + 4 * t + r;
    const float ax = Xa[0], ay = Xa[K], az = Xa[2 * K];
    const float bx = Xa[2], by = Xa[K + 2], bz = Xa[2 * K + 2];
    float* ra = S + 3 * K + (8 * t + 4 * r) * (t + 1);  // row_off(4 t + r)
#pragma unroll 1
    for (int c = 0; c < t; c++) {
      const float4 X = *reinterpret_cast<const float4*>(S + 4 * c);
      const float4 Y = *reinterpret_cast<const float4*>(S + K + 4 * c);
      const float4 Z = *reinterpret_cast<const float4*>(S + 2 * K + 4 * c);
      const float2 x0 = make_float2(X.x, X.y), x1 = make_float2(X.z, X.w);
      const float2 y0 = make_float2(Y.x, Y.y), y1 = make_float2(Y.z, Y.w);
      const float2 z0 = make_float2(Z.x, Z.y), z1 = make_float2(Z.z, Z.w);
      const float2 e0 = entry_pair<KT>(kf, rf, sqdist2(sub2(ax, x0), sub2(ay, y0), sub2(az, z0)));
      const float2 e1 = entry_pair<KT>(kf, rf, sqdist2(sub2(ax, x1), sub2(ay, y1), sub2(az, z1)));
      const float2 e2 = entry_pair<KT>(kf, rf, sqdist2(sub2(bx, x0), sub2(by, y0), sub2(bz, z0)));
      const float2 e3 = entry_pair<KT>(kf, rf, sqdist2(sub2(bx, x1), sub2(by, y1), sub2(bz, z1)));
      *reinterpret_cast<float4*>(ra + 4 * c) = make_float4(e0.x, e0.y, e1.x, e1.y);
      *reinterpret_cast<float4*>(ra + 8 * (t + 1) + 4 * c) = make_float4(e2.x, e2.y, e3.x, e3.y);
    }
  }
  constexpr int TB = K / 4 > 1 ? 2 : 1;  // diagonal blocks per step
#pragma unroll 1
  for (int t = 0; 4 * t < k; t += TB) {
    const int t1 = TB == 2 && 4 * (t + 1) < K ? t + 1 : t;  // K = 12: the last one twice
    const float4 X0 = *reinterpret_cast<const float4*>(S + 4 * t);
    const float4 Y0 = *reinterpret_cast<const float4*>(S + K + 4 * t);
    const float4 Z0 = *reinterpret_cast<const float4*>(S + 2 * K + 4 * t);
    const float4 X1 = *reinterpret_cast<const float4*>(S + 4 * t1);
    const float4 Y1 = *reinterpret_cast<const float4*>(S + K + 4 * t1);
    const float4 Z1 = *reinterpret_cast<const float4*>(S + 2 * K + 4 * t1);
    auto at = [&](float u0, float w0, float u1, float w1) { return make_float2(u0 - w0, u1 - w1); };
    // lane 0: (1, 0) (2, 0) (3, 0); lane 1: (2, 1) (3, 1) (3, 2); then (2 r, i) (2 r + 1, i)
#define GGP_PICK(u, w)                                                              \
  sqdist2(at(r ? X0.u : X0.w, r ? X0.GGP_V : X0.x, r ? X1.u : X1.w, r ? X1.GGP_V : X1.x), \
          at(r ? Y0.u : Y0.w, r ? Y0.GGP_V : Y0.x, r ? Y1.u : Y1.w, r ? Y1.GGP_V : Y1.x), \
          at(r ? Z0.u : Z0.w, r ? Z0.GGP_V : Z0.x, r ? Z1.u : Z1.w, r ? Z1.GGP_V : Z1.x))
#define GGP_V y
    const float2 e0 = entry_pair<KT>(kf, rf, GGP_PICK(z, y));
    const float2 e1 = entry_pair<KT>(kf, rf, GGP_PICK(w, z));
#undef GGP_V
#define GGP_V z
    const float2 e2 = entry_pair<KT>(kf, rf, GGP_PICK(w, w));
#undef GGP_V
#undef GGP_PICK
    const float2 q0 = entry_pair<KT>(
        kf, rf, sqdist2(at(r ? X0.z : X0.x, xq.x, r ? X1.z : X1.x, xq.x),
                        at(r ? Y0.z : Y0.x, xq.y, r ? Y1.z : Y1.x, xq.y),
                        at(r ? Z0.z : Z0.x, xq.z, r ? Z1.z : Z1.x, xq.z)));
    const float2 q1 = entry_pair<KT>(
        kf, rf, sqdist2(at(r ? X0.w : X0.y, xq.x, r ? X1.w : X1.y, xq.x),
                        at(r ? Y0.w : Y0.y, xq.y, r ? Y1.w : Y1.y, xq.y),
                        at(r ? Z0.w : Z0.y, xq.z, r ? Z1.w : Z1.y, xq.z)));
#pragma unroll
    for (int h = 0; h < TB; h++) {
      const int tb = h ? t1 : t, len = 4 * (tb + 1);
      float* rd = S + 3 * K + 8 * tb * (tb + 1) + 4 * tb;  // row 4 tb, column 4 tb
      rd[r ? 2 * len + 1 : len] = h ? e0.y : e0.x;
      rd[r ? 3 * len + 1 : 2 * len] = h ? e1.y : e1.x;
      rd[r ? 3 * len + 2 : 3 * len] = h ? e2.y : e2.x;
      rd[2 * r * (len + 1)] = h ? q0.y : q0.x;
      rd[(2 * r + 1) * (len + 1)] = h ? q1.y : q1.x;
    }
  }
  __syncwarp();
  // the lane's rows into registers; their diagonal place holds the value with
  // the point
  float2 yv[R / 2];  // slots 2 t (x) and 2 t + 1 (y)
  static_for<0, R>([&](auto Sc) {
    constexpr int s = decltype(Sc)::value;
#pragma unroll
    for (int c = 0; c <= s / 2; c++) {
      const float4 q = *reinterpret_cast<const float4*>(
          S + PL::row_off(2 * s) + 4 * (s / 2 + 1) * r + 4 * c);
      f.A[PF::ap(s, 2 * c)] = make_float2(q.x, q.y);
      if (2 * c + 1 <= s) f.A[PF::ap(s, 2 * c + 1 <= s ? 2 * c + 1 : s)] = make_float2(q.z, q.w);
    }
    const float e = r ? f.A[PF::ap(s, s)].y : f.A[PF::ap(s, s)].x;
    if (s & 1) yv[s / 2].y = e; else yv[s / 2].x = e;
  });
  __syncwarp();
  auto yown = [&](auto Sc) -> float& {
    constexpr int s = decltype(Sc)::value;
    return s & 1 ? yv[s / 2].y : yv[s / 2].x;
  };
  // -M and m
  const float e0i = __shfl_sync(full, yv[0].x, 0, 2);  // gamma_0i or -kappa_0i
  f.varw = inc ? 2.0f * (e0i + nug) : k0;
  // gamma_a0 of every row, negated, in the rows' (still unused) place
  static_for<0, R>([&](auto Sc) {
    constexpr int s = decltype(Sc)::value;
    S[PL::row_off(0) + 2 * s + r] = -f.A[PF::ap(s, 0)].x;
  });
  __syncwarp();
  if (inc) {
    float2 g0[R];
#pragma unroll
    for (int c = 0; c < K / 4; c++) {
      const float4 q = *reinterpret_cast<const float4*>(S + PL::row_off(0) + 4 * c);
      g0[2 * c] = make_float2(q.x, q.y);
      g0[2 * c + 1] = make_float2(q.z, q.w);
    }
    static_for<0, R>([&](auto Sc) {
      constexpr int s = decltype(Sc)::value;
      const float ea0 = f.A[PF::ap(s, 0)].x;
      // -(((ea0 + ec0) - e) + nug); the columns past the diagonal are not used
#pragma unroll
      for (int c = 0; c <= s; c++)
        f.A[PF::ap(s, c)] = __fadd2_rn(
            __fadd2_rn(f.A[PF::ap(s, c)], __fadd2_rn(two(-ea0), g0[c])), two(-nug));
      const float en = ea0 + nug;
      float2& d = f.A[PF::ap(s, s)];
      const float dd = -2.0f * en;
      if (r) d.y = dd; else d.x = dd;
      if (s > 0 || r) f.A[PF::ap(s, 0)].x = en;  // column 0
      float& y = yown(Sc);
      y = ((ea0 + e0i) - y) + nug;
    });
    if (r == 0) {  // row 0
      f.A[0].x = -k0;
      yv[0].x = -(e0i + nug);
    }
  } else {
    static_for<0, R>([&](auto Sc) {
      constexpr int s = decltype(Sc)::value;
      float2& d = f.A[PF::ap(s, s)];
      if (r) d.y = -k0; else d.x = -k0;
      float& y = yown(Sc);
      y = -y;
    });
  }
  static_for<0, R>([&](auto Sc) {  // rows past k: identity padding
    constexpr int s = decltype(Sc)::value;
    if (2 * s + 1 >= k) {
      const bool pad = 2 * s + r >= k;
#pragma unroll
      for (int c = 0; c <= s; c++)
        if (pad) f.A[PF::ap(s, c)] = make_float2(c == s && !r ? -1.0f : 0.0f, c == s && r ? -1.0f : 0.0f);
      if (pad) yown(Sc) = 0.0f;
    }
  });
  __syncwarp();  // gamma_a0 is read
  DF s2{f.varw, 0.0f};
  bool clamped = false;
  float max_ratio = 1.0f;
  const float pfloor = fmaxf(kPdFloor * k0, kPivotMin);
  static_for<0, K>([&](auto Jc) {
    constexpr int j = decltype(Jc)::value;
    constexpr int sj = j / 2, rj = j % 2;
    float2 Lj[(j + 3) / 4 * 2 + 2];
#pragma unroll
    for (int c = 0; c < (j + 3) / 4; c++) {
      const float4 q = *reinterpret_cast<const float4*>(S + PL::row_off(j) + 4 * c);
      Lj[2 * c] = make_float2(q.x, q.y);
      Lj[2 * c + 1] = make_float2(q.z, q.w);
    }
    float nt[R];  // -(M_aj - sum_m L_am L_jm) of the lane's rows
    static_for<sj, R>([&](auto Sc) {
      constexpr int s = decltype(Sc)::value;
      const float2 m0 = f.A[PF::ap(s, sj)];
      float2 acc = make_float2(rj ? m0.y : m0.x, 0.0f);
#pragma unroll
      for (int c = 0; c < j / 4 * 2; c++) acc = __ffma2_rn(f.A[PF::ap(s, c)], Lj[c], acc);
#pragma unroll
      for (int m = j / 4 * 4; m < j; m++)
        acc.x = m & 1 ? __fmaf_rn(f.A[PF::ap(s, m / 2)].y, Lj[m / 2].y, acc.x)
                      : __fmaf_rn(f.A[PF::ap(s, m / 2)].x, Lj[m / 2].x, acc.x);
      nt[s] = acc.x + acc.y;
    });
    float piv = -__shfl_sync(full, nt[sj], rj, 2);
    if (!(piv > pfloor)) {
      piv = pfloor;
      clamped = true;
    }
    const float inv = rcp_newton(sqrt_newton(piv));
    const float mjj = -(rj ? f.A[PF::ap(sj, sj)].y : f.A[PF::ap(sj, sj)].x);
    if (r == rj) max_ratio = fmaxf(max_ratio, mjj * inv * inv);
    const float yj = __shfl_sync(full, yown(std::integral_constant<int, sj>{}), rj, 2) * inv;
    s2 = df_sub_square(s2, yj);
    if (rj) f.b[sj].y = yj; else f.b[sj].x = yj;
    static_for<sj, R>([&](auto Sc) {  // rows up to j: not used any more
      constexpr int s = decltype(Sc)::value;
      const float l = nt[s] * -inv;
      if (rj) f.A[PF::ap(s, sj)].y = l; else f.A[PF::ap(s, sj)].x = l;
      float& y = yown(Sc);
      y = __fmaf_rn(l, -yj, y);
    });
    S[PL::row_off(j) + j] = inv;
    if constexpr (j == K * 3 / 4) late();
    if constexpr (j + 1 < K) {  // row j + 1 is complete
      constexpr int sn = (j + 1) / 2;
      if (r == (j + 1) % 2) {
#pragma unroll
        for (int c = 0; c < j / 4 + 1; c++) {
          const float2 u = f.A[PF::ap(sn, 2 * c)];
          const float2 w = 2 * c + 1 <= sn ? f.A[PF::ap(sn, 2 * c + 1 <= sn ? 2 * c + 1 : sn)]
                                           : make_float2(0.0f, 0.0f);
          *reinterpret_cast<float4*>(S + PL::row_off(j + 1) + 4 * c) =
              make_float4(u.x, u.y, w.x, w.y);
        }
      }
      __syncwarp();
    }
  });
  float sig2 = s2.hi + s2.lo;
  if (!(sig2 > pfloor)) {
    sig2 = pfloor;
    clamped = true;
  }
  f.clamped = clamped;
  f.max_ratio = fmaxf(max_ratio, __shfl_xor_sync(full, max_ratio, 1));
  f.sigma = sqrtf(sig2);
  done();
  // beta = L^-T y, last entry first, on both lanes
  __syncwarp();
  pair_back_solve<K>(S, f.b);
  // increment form: b_0 = 1 + beta_0 - sum_{a>=1} beta_a (padding entries are zero)
  float sb = 0.0f;
#pragma unroll
  for (int a = 1; a < K; a++) sb += f.weight(a);
  if (inc) f.b[0].x = (1.0f + f.b[0].x) - sb;
  f.finite = isfinite(sb) && isfinite(f.b[0].x);  // a non-finite weight makes the sum so
}

// Whether the row must be recomputed in FP64 (rescue.cuh), the same on both
// lanes: a floored pivot or sigma^2, a row-error estimate above the kernel's
// threshold, or a non-finite weight or sigma.
template <int K>
__device__ __forceinline__ bool pair_needs_rescue(const PairFactor<K>& f, const KernF& kf) {
  return f.clamped || row_error_too_large(f.max_ratio, f.varw, f.sigma, kf) || !isfinite(f.sigma) ||
         !f.finite;
}

// The weight of the lane's slot s.
template <int K>
__device__ __forceinline__ float pair_own(const float2 (&b)[K / 2], int r, int s) {
  return r ? b[s].y : b[s].x;
}

// The field at the neighbours of the lane's slots.  LEVEL: v is written level
// by level in the same launch.
template <int K, bool LEVEL>
__device__ __forceinline__ void pair_gather(float (&vv)[K / 2], int r,
                                            const int32_t* __restrict__ row, const float* v,
                                            uint64_t pol) {
#pragma unroll
  for (int s = 0; s < K / 2; s++) {
    const int2 c = __ldg(reinterpret_cast<const int2*>(row) + s);
    vv[s] = LEVEL ? ld_level_f(v + (r ? c.y : c.x), pol) : ld_keep_f(v + (r ? c.y : c.x), pol);
  }
}

// sum_a b_a v[c_a] in the stored sweeps' summation order (sweepsync.cuh):
// lane 0 holds the even entries of every slice, lane 1 the odd ones, which are
// the two alternating accumulators.
template <int K>
__device__ __forceinline__ float pair_dot(const float2 (&b)[K / 2], const float (&vv)[K / 2],
                                          int r) {
  constexpr int LANES = gen_lanes(K), HS = K / LANES / 2;
  float part[LANES];
#pragma unroll
  for (int h = 0; h < LANES; h++) {
    float acc = 0.0f;
#pragma unroll
    for (int u = 0; u < HS; u++) acc = fmaf(pair_own<K>(b, r, h * HS + u), vv[h * HS + u], acc);
    part[h] = acc + __shfl_xor_sync(0xffffffffu, acc, 1);
  }
  if (LANES == 4) return (part[0] + part[2 % LANES]) + (part[1 % LANES] + part[3 % LANES]);
  if (LANES == 2) return part[0] + part[1 % LANES];
  return part[0];
}

// The rows of the warp's points with `need` set recomputed in FP64, one at a
// time by the whole warp (warp_row_factor64); both lanes of such a point
// receive its b (zero past k), sigma and floor flag.  A collective; Sw: the
// shared memory of the warp's points, which is overwritten.
template <int K, int KT>
__device__ __forceinline__ void pair_rescue(PairFactor<K>& f, bool need, float* Sw,
                                            const float4* __restrict__ xs, const int32_t* row,
                                            int k, float4 xq, const KernF& kf) {
  static_assert(16 * PairLayout<K>::kStride * sizeof(float) >= K * (K + 1) * sizeof(double), "");
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  unsigned m = __ballot_sync(full, need) & 0x55555555u;
  while (m) {
    const int src = __ffs(m) - 1;
    m &= m - 1;
    const int32_t* rw = reinterpret_cast<const int32_t*>(
        __shfl_sync(full, reinterpret_cast<unsigned long long>(row), src));
    float4 q;
    q.x = __shfl_sync(full, xq.x, src);
    q.y = __shfl_sync(full, xq.y, src);
    q.z = __shfl_sync(full, xq.z, src);
    q.w = 0.0f;
    const WarpRow64 w = warp_row_factor64<K, KT>(xs, rw, k, q, kf, reinterpret_cast<double*>(Sw));
    if (lane < K) Sw[lane] = lane < k ? (float)w.b : 0.0f;
    __syncwarp();
    if ((lane & ~1) == src) {
#pragma unroll
      for (int c = 0; c < K / 2; c++) f.b[c] = make_float2(Sw[2 * c], Sw[2 * c + 1]);
      f.sigma = (float)w.sigma;
      f.clamped = w.clamped;
    }
    __syncwarp();
  }
}

// kappa and d kappa / d lengthscale of two squared distances: the operations of
// kappa_dkappa_d2 on packed pairs.
struct DPair {
  float2 k, l;
};

template <int KT>
__device__ __forceinline__ DPair dentry_pair(const KernF& kf, float2 d2) {
  const float2 s2 = two(kf.s2), il = two(kf.inv_ell);
  if (KT == GRAPHGP_MATERN12) {
    const float2 r = sqrt_pair(d2), a = __fmul2_rn(r, il);
    const float2 k = __fmul2_rn(s2, make_float2(expf(-a.x), expf(-a.y)));
    return DPair{k, __fmul2_rn(__fmul2_rn(__fmul2_rn(k, r), il), il)};
  }
  const float2 a = arg_pair<KT>(kf, d2);
  const float2 e = make_float2(expf(-a.x), expf(-a.y));
  if (KT == GRAPHGP_SQEXP) {
    const float2 k = __fmul2_rn(s2, e);
    return DPair{k, __fmul2_rn(__fmul2_rn(__fmul2_rn(__fmul2_rn(k, d2), il), il), il)};
  }
  const float2 p = __fadd2_rn(two(1.0f), a), saa = __fmul2_rn(__fmul2_rn(s2, a), a);
  if (KT == GRAPHGP_MATERN32)
    return DPair{__fmul2_rn(__fmul2_rn(s2, p), e), __fmul2_rn(__fmul2_rn(saa, e), il)};
  const float2 q = __ffma2_rn(__fmul2_rn(a, a), two(1.0f / 3.0f), p);
  return DPair{__fmul2_rn(__fmul2_rn(s2, q), e),
               __fmul2_rn(__fmul2_rn(__fmul2_rn(__fmul2_rn(saa, p), e), il), two(1.0f / 3.0f))};
}

// Running sums of one row of Kbar against both derivatives, one value at a
// time in the order of the columns.
struct RowTheta {
  float s, l;
  __device__ __forceinline__ void add(float kb, float k, float dl, float inv_s2) {
    s = __fmaf_rn(__fmul_rn(kb, k), inv_s2, s);
    l = __fmaf_rn(kb, dl, l);
  }
};

// The per-row factor backward, after pair_factor left the lane's rows of L in
// f and all of them, with the coordinates, in S: g = K_cc^-1 (alpha v_c), then
// Kbar against dkappa/dtheta: the pair (a, c), c < a, takes Kbar_ac + Kbar_ca =
// (-g_a b_c + sbar b_a b_c) + (-g_c b_a + sbar b_c b_a), the diagonal -g_a b_a +
// sbar b_a^2, (a, i) g_a - 2 sbar b_a, and Kbar_ii = sbar.  These terms cancel to
// a small part of their size, so their order is fixed: each row's sum in FP32
// over its columns in ascending order and (a, i) last (at most k + 1 terms),
// then added to the FP64 totals.  A lane takes its own rows, two at a time,
// four columns per step; in the last step of a row the point stands in the
// column after the diagonal's.  (Sharing a diagonal block's pairs between the
// lanes and keeping two partial sums per row is 10 % faster but moves the
// sigma2 component, the worst conditioned, by 1e-6 of the gradient and more.)
// Every lane of the warp must call this; `act` says whether the point counts.
// S's rows of L are overwritten.
template <int K, int KT>
__device__ __forceinline__ void pair_row_backward(const PairFactor<K>& f, float* S, int r, int k,
                                                  const KernF& kf, float4 xq,
                                                  const float (&vv)[K / 2], float alpha,
                                                  float sbar, bool act, double& tl, double& ts,
                                                  double& tn) {
  using PL = PairLayout<K>;
  using PF = PairFactor<K>;
  constexpr int R = K / 2;
  const unsigned full = 0xffffffffu;
  const float inv_s2 = 1.0f / kf.s2;
  float g[R];
#pragma unroll
  for (int s = 0; s < R; s++) g[s] = 2 * s + r < k ? alpha * vv[s] : 0.0f;
  const float r0 = __shfl_sync(full, g[0], 0, 2);
  if (f.inc) {
#pragma unroll
    for (int s = 0; s < R; s++)
      if (2 * s + r >= 1 && 2 * s + r < k) g[s] -= r0;
  }
  float2 z[R];
  static_for<0, K>([&](auto Jc) {
    constexpr int j = decltype(Jc)::value;
    constexpr int sj = j / 2, rj = j % 2;
    const float zj = __shfl_sync(full, g[sj], rj, 2) * S[PL::row_off(j) + j];
    if (rj) z[sj].y = zj; else z[sj].x = zj;
    if (rj == 0) {  // row j + 1 is lane 1's
      const float t = __fmaf_rn(f.A[PF::ap(sj, sj)].x, -zj, g[sj]);
      if (r) g[sj] = t;
    }
    static_for<sj + 1, R>([&](auto Sc) {
      constexpr int s = decltype(Sc)::value;
      const float2 l = f.A[PF::ap(s, sj)];
      g[s] = __fmaf_rn(rj ? l.y : l.x, -zj, g[s]);
    });
  });
  pair_back_solve<K>(S, z);
  float sg = 0.0f;
#pragma unroll
  for (int a = 1; a < K; a++) sg += a & 1 ? z[a / 2].y : z[a / 2].x;
  if (f.inc) z[0].x -= sg;
  // g and b in the place of L's rows; the solves are done on both lanes
  __syncwarp();
  float* G = S + 3 * K;
  float* B = G + K;
#pragma unroll
  for (int c = 0; c < K / 4; c++) {
    const float2 u = r ? f.b[2 * c] : z[2 * c], w = r ? f.b[2 * c + 1] : z[2 * c + 1];
    *reinterpret_cast<float4*>((r ? B : G) + 4 * c) = make_float4(u.x, u.y, w.x, w.y);
  }
  __syncwarp();
  double dl = 0.0, ds = r ? 0.0 : (double)sbar, dn = ds;  // Kbar_ii = sbar
#pragma unroll 1
  for (int t = 0; 4 * t < k; t++) {
    float ng[2], ba[2], sba[2], px[2], py[2], pz[2];
    RowTheta th[2];
    float kaa[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const int a = 4 * t + 2 * h + r;
      ng[h] = -G[a];
      ba[h] = B[a];
      sba[h] = __fmul_rn(sbar, ba[h]);
      px[h] = S[a];
      py[h] = S[K + a];
      pz[h] = S[2 * K + a];
      kaa[h] = __fmaf_rn(sba[h], ba[h], __fmul_rn(ng[h], ba[h]));
      th[h] = RowTheta{kaa[h], 0.0f};
    }
#pragma unroll 1
    for (int c = 0; c <= t; c++) {
      float4 X = *reinterpret_cast<const float4*>(S + 4 * c);
      float4 Y = *reinterpret_cast<const float4*>(S + K + 4 * c);
      float4 Z = *reinterpret_cast<const float4*>(S + 2 * K + 4 * c);
      const float4 Gc = *reinterpret_cast<const float4*>(G + 4 * c);
      const float4 Bc = *reinterpret_cast<const float4*>(B + 4 * c);
      const float2 b0 = make_float2(Bc.x, Bc.y), b1 = make_float2(Bc.z, Bc.w);
      const float2 g0 = make_float2(-Gc.x, -Gc.y), g1 = make_float2(-Gc.z, -Gc.w);
      const float2 s0 = __fmul2_rn(two(sbar), b0), s1 = __fmul2_rn(two(sbar), b1);
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const int q = c == t ? 2 * h + r : 4;  // column of the diagonal in this step
        auto at = [&](float4 u, float pt, int i) {
          const float x = i == 0 ? u.x : i == 1 ? u.y : i == 2 ? u.z : u.w;
          return i == q ? pt : x;
        };
        auto val = [&](int i) {
          return dentry_pair<KT>(
              kf, sqdist2(sub2(px[h], make_float2(at(X, xq.x, i), at(X, xq.x, i + 1))),
                          sub2(py[h], make_float2(at(Y, xq.y, i), at(Y, xq.y, i + 1))),
                          sub2(pz[h], make_float2(at(Z, xq.z, i), at(Z, xq.z, i + 1)))));
        };
        auto cot = [&](float2 gc, float2 bc, float2 sc) {
          return __fadd2_rn(
              __ffma2_rn(two(sba[h]), bc, __fmul2_rn(two(ng[h]), bc)),
              __ffma2_rn(sc, two(ba[h]), __fmul2_rn(gc, two(ba[h]))));
        };
        const float2 k0 = cot(g0, b0, s0), k1 = cot(g1, b1, s1);
        const float kci = __fmaf_rn(-2.0f * sbar, ba[h], -ng[h]);
        const DPair d0 = val(0), d1 = val(2);
        auto pick = [&](float kb, int i) { return i < q ? kb : (i == q ? kci : 0.0f); };
        th[h].add(pick(k0.x, 0), d0.k.x, d0.l.x, inv_s2);
        th[h].add(pick(k0.y, 1), d0.k.y, d0.l.y, inv_s2);
        th[h].add(pick(k1.x, 2), d1.k.x, d1.l.x, inv_s2);
        th[h].add(pick(k1.y, 3), d1.k.y, d1.l.y, inv_s2);
      }
    }
#pragma unroll
    for (int h = 0; h < 2; h++)
      if (4 * t + 2 * h + r < k) {
        dl += th[h].l;
        ds += th[h].s;
        dn += kaa[h];
      }
  }
  if (act) {
    tl += dl;
    ts += ds;
    tn += dn;
  }
}

}  // namespace ggp
