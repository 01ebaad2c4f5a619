// Per-point conditional factor for 16 < k <= 32: eight lanes per point.
//
// The arithmetic and its order are those of pointpair.cuh (increment or
// covariance form, left-looking Cholesky with two accumulators, compensated
// sigma^2, backward sweep); only the split differs.  Lane r of a point's eight
// owns the rows a = 8 s + r of M (slot s, K / 8 slots), as packed pairs of
// columns in registers; finished rows of L are published in shared memory.  K
// is 24 or 32; row lengths kp = 20 .. 32 of the stored arrays need not equal
// it.
//
// Why eight lanes: a warp covers four points, so what every column costs
// whatever the number of lanes (broadcasts, pivot, root, reciprocal, the
// compensated sum: about 35 instructions, 32 times) is shared by four points,
// and a lane's rows take 80 registers at K = 32.  With one warp per point each
// covariance value was computed on both sides of the diagonal and a step of
// the Cholesky used half its lanes on average.  Measured (2^20 uniform points,
// k = 32, squared exponential, one warp -> eight lanes per point, each call
// with its dense block): factor 8.9 -> 3.4 ms; factor + NLL + gradient 27.6 ->
// 12.1 ms.
#pragma once

#include "pointpair.cuh"

namespace ggp {

// Shared memory of one point: x[K], y[K], z[K], the rows of L as in
// PairLayout, then two vectors (weights, field or cotangents).
template <int K>
struct OctLayout {
  static constexpr int R = K / 8;  // rows per lane
  static __host__ __device__ constexpr int row_off(int a) {
    return 3 * K + 8 * (a / 4) * (a / 4 + 1) + 4 * (a % 4) * (a / 4 + 1);
  }
  static constexpr int kVecB = row_off(K), kVecV = kVecB + K;
  static constexpr int kUsed = kVecV + K;
  static constexpr int kStride = kUsed / 4 % 2 ? kUsed : kUsed + 4;
  static constexpr int kPoints = kPairThreads / 8;  // points per block
  static constexpr size_t kBytes = (size_t)kPoints * kStride * sizeof(float);
  static constexpr int kBlocks = K > 24 ? 3 : 4;  // per SM: 168 or 128 registers per thread
};

template <int K>
inline unsigned oct_grid(int64_t npts) {
  const int64_t blocks = (npts + OctLayout<K>::kPoints - 1) / OctLayout<K>::kPoints;
  const int64_t most = (int64_t)OctLayout<K>::kBlocks * num_sms();
  return (unsigned)(blocks < most ? blocks : most);
}

template <int K>
struct OctFactor {
  static constexpr int R = K / 8;
  float2 A[2 * R * (R + 1)];  // slot s, columns 2c, 2c + 1 at ap(s, c)
  float b[R];                 // the lane's weights (zero past k)
  float sigma, max_ratio, varw;
  bool clamped, inc, finite;
  static __host__ __device__ constexpr int ap(int s, int c) { return 2 * s * (s + 1) + c; }
};

// Gathers the neighbour coordinates of a row into the point's shared memory,
// one chunk of four per lane (entries past kp: index 0).
template <int K>
__device__ __forceinline__ void oct_stage(float* S, int r, const float4* __restrict__ xs,
                                          const int32_t* __restrict__ row, int kp) {
  __syncwarp();  // earlier readers of S are done
  if (4 * r < K) {
    const int4 n = 4 * r < kp ? __ldg(reinterpret_cast<const int4*>(row) + r) : make_int4(0, 0, 0, 0);
    const float4 x0 = __ldg(xs + n.x), x1 = __ldg(xs + n.y), x2 = __ldg(xs + n.z),
                 x3 = __ldg(xs + n.w);
    *reinterpret_cast<float4*>(S + 4 * r) = make_float4(x0.x, x1.x, x2.x, x3.x);
    *reinterpret_cast<float4*>(S + K + 4 * r) = make_float4(x0.y, x1.y, x2.y, x3.y);
    *reinterpret_cast<float4*>(S + 2 * K + 4 * r) = make_float4(x0.z, x1.z, x2.z, x3.z);
  }
  __syncwarp();
}

// y <- L^-T y with the rows of L in shared memory, last entry first; the lane
// holds the entries of its slots.
template <int K>
__device__ __forceinline__ void oct_back_solve(const float* S, int r, float (&y)[K / 8]) {
  static_for<0, K>([&](auto Jr) {
    constexpr int j = K - 1 - decltype(Jr)::value;
    constexpr int sj = j / 8, rj = j % 8;
    const float* Lj = S + OctLayout<K>::row_off(j);
    const float bj = __shfl_sync(0xffffffffu, y[sj] * Lj[j], rj, 8);
#pragma unroll
    for (int s = 0; s < sj; s++) y[s] = __fmaf_rn(Lj[8 * s + r], -bj, y[s]);
    const float l = Lj[8 * sj + min(r, rj)];
    y[sj] = r < rj ? __fmaf_rn(l, -bj, y[sj]) : (r == rj ? bj : y[sj]);
  });
}

// x[1] + x[2] + .. + x[K - 1] in order, entry a on lane a % 8, slot a / 8.
template <int K>
__device__ __forceinline__ float oct_sum_from_1(const float (&x)[K / 8]) {
  float sum = 0.0f;
#pragma unroll
  for (int a = 1; a < K; a++) sum += __shfl_sync(0xffffffffu, x[a / 8], a % 8, 8);
  return sum;
}

template <int K, int KT>
__device__ __forceinline__ void oct_factor(OctFactor<K>& f, float* S, int r, int k,
                                           const KernF& kf, float4 xq) {
  using OL = OctLayout<K>;
  using OF = OctFactor<K>;
  constexpr int R = K / 8;
  const unsigned full = 0xffffffffu;
  const float k0 = kf.s2 + kf.nug, nug = kf.nug;
  const float g0i = gamma_at<KT>(
      kf, cov_arg<KT>(kf, sqdist(make_float4(S[0], S[K], S[2 * K], 0.0f), xq)));
  const bool inc = g0i < 0.5f * kf.s2;
  f.inc = inc;
  const RowForm rf{inc ? cov_switch<KT>() : -1.0f, inc ? 1.0f : 0.0f};
  // covariance values into the rows' place: the lane's row 8 s + r against the
  // columns left of its 8 x 8 diagonal block, eight at a time
#pragma unroll 1
  for (int s = 1; 8 * s < k; s++) {
    const int a = 8 * s + r;
    const float ax = S[a], ay = S[K + a], az = S[2 * K + a];
    float* ra = S + 3 * K + 8 * (a / 4) * (a / 4 + 1) + 4 * (a % 4) * (a / 4 + 1);
#pragma unroll 1
    for (int c = 0; c < s; c++) {
      const float4 X0 = *reinterpret_cast<const float4*>(S + 8 * c);
      const float4 X1 = *reinterpret_cast<const float4*>(S + 8 * c + 4);
      const float4 Y0 = *reinterpret_cast<const float4*>(S + K + 8 * c);
      const float4 Y1 = *reinterpret_cast<const float4*>(S + K + 8 * c + 4);
      const float4 Z0 = *reinterpret_cast<const float4*>(S + 2 * K + 8 * c);
      const float4 Z1 = *reinterpret_cast<const float4*>(S + 2 * K + 8 * c + 4);
      auto val = [&](float2 x, float2 y, float2 z) {
        return entry_pair<KT>(kf, rf, sqdist2(sub2(ax, x), sub2(ay, y), sub2(az, z)));
      };
      const float2 e0 = val(make_float2(X0.x, X0.y), make_float2(Y0.x, Y0.y), make_float2(Z0.x, Z0.y));
      const float2 e1 = val(make_float2(X0.z, X0.w), make_float2(Y0.z, Y0.w), make_float2(Z0.z, Z0.w));
      const float2 e2 = val(make_float2(X1.x, X1.y), make_float2(Y1.x, Y1.y), make_float2(Z1.x, Z1.y));
      const float2 e3 = val(make_float2(X1.z, X1.w), make_float2(Y1.z, Y1.w), make_float2(Z1.z, Z1.w));
      *reinterpret_cast<float4*>(ra + 8 * c) = make_float4(e0.x, e0.y, e1.x, e1.y);
      *reinterpret_cast<float4*>(ra + 8 * c + 4) = make_float4(e2.x, e2.y, e3.x, e3.y);
    }
  }
  // the diagonal blocks, two at a time (x and y of the packed values): of a
  // block's 28 pairs the lane takes (r, r + d mod 8), d = 1, 2, 3; of the four
  // pairs (u, u + 4) lanes 0..3 take the first block's, lanes 4..7 the
  // second's; and each block's value of row r with the point, which is put in
  // the row's diagonal place
#pragma unroll 1
  for (int s = 0; 8 * s < k; s += 2) {
    const int s1 = 8 * (s + 1) < K ? s + 1 : s;  // K = 24: the last one twice
    const int o0 = 8 * s, o1 = 8 * s1;
    auto dist = [&](int u0, int w0, int u1, int w1) {
      return sqdist2(make_float2(S[u0] - S[w0], S[u1] - S[w1]),
                     make_float2(S[K + u0] - S[K + w0], S[K + u1] - S[K + w1]),
                     make_float2(S[2 * K + u0] - S[2 * K + w0], S[2 * K + u1] - S[2 * K + w1]));
    };
    auto put = [&](int a, int c, float e) {
      S[3 * K + 8 * (a / 4) * (a / 4 + 1) + 4 * (a % 4) * (a / 4 + 1) + c] = e;
    };
#pragma unroll
    for (int d = 1; d < 4; d++) {
      const int w = (r + d) & 7, hi = max(r, w), lo = min(r, w);
      const float2 e = entry_pair<KT>(kf, rf, dist(o0 + hi, o0 + lo, o1 + hi, o1 + lo));
      put(o0 + hi, o0 + lo, e.x);
      put(o1 + hi, o1 + lo, e.y);
    }
    const int o4 = r < 4 ? o0 : o1, u = r & 3;
    const float2 q0 = make_float2(S[o4 + u + 4] - S[o4 + u], S[o0 + r] - xq.x);
    const float2 q1 = make_float2(S[K + o4 + u + 4] - S[K + o4 + u], S[K + o0 + r] - xq.y);
    const float2 q2 = make_float2(S[2 * K + o4 + u + 4] - S[2 * K + o4 + u], S[2 * K + o0 + r] - xq.z);
    const float2 e4 = entry_pair<KT>(kf, rf, sqdist2(q0, q1, q2));
    put(o4 + u + 4, o4 + u, e4.x);
    put(o0 + r, o0 + r, e4.y);
    const float2 e5 = entry_pair<KT>(
        kf, rf, sqdist2(two(S[o1 + r] - xq.x), two(S[K + o1 + r] - xq.y), two(S[2 * K + o1 + r] - xq.z)));
    put(o1 + r, o1 + r, e5.x);
  }
  __syncwarp();
  // the lane's rows into registers; m from the diagonal place
  float yv[R];
  static_for<0, R>([&](auto Sc) {
    constexpr int s = decltype(Sc)::value;
    // row 8 s + r: its padded length is 8 s + 4 for r < 4, 8 s + 8 above
    const float* ra = S + OL::row_off(8 * s) +
                      (r < 4 ? r * (8 * s + 4) : 4 * (8 * s + 4) + (r - 4) * (8 * s + 8));
#pragma unroll
    for (int c = 0; c <= 2 * s + 1; c++) {
      float4 q = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (c <= 2 * s || r >= 4) q = *reinterpret_cast<const float4*>(ra + 4 * c);
      f.A[OF::ap(s, 2 * c)] = make_float2(q.x, q.y);
      f.A[OF::ap(s, 2 * c + 1)] = make_float2(q.z, q.w);
    }
    yv[s] = ra[8 * s + r];
  });
  const float e0i = __shfl_sync(full, yv[0], 0, 8);  // gamma_0i or -kappa_0i
  f.varw = inc ? 2.0f * (e0i + nug) : k0;
  static_for<0, R>([&](auto Sc) {  // gamma_a0 of every row, negated
    constexpr int s = decltype(Sc)::value;
    S[OL::kVecB + 8 * s + r] = -f.A[OF::ap(s, 0)].x;
  });
  __syncwarp();
  // sets the diagonal entry of slot s
  auto set_diag = [&](auto Sc, float v) {
    constexpr int s = decltype(Sc)::value;
#pragma unroll
    for (int c = 0; c < 4; c++) {
      float2& d = f.A[OF::ap(s, 4 * s + c)];
      if (r == 2 * c) d.x = v;
      if (r == 2 * c + 1) d.y = v;
    }
  };
  if (inc) {
    static_for<0, R>([&](auto Sc) {
      constexpr int s = decltype(Sc)::value;
      const float ea0 = f.A[OF::ap(s, 0)].x;
      // -(((ea0 + ec0) - e) + nug); the columns past the diagonal are not used
#pragma unroll
      for (int c = 0; c <= 2 * s + 1; c++) {
        const float4 q = *reinterpret_cast<const float4*>(S + OL::kVecB + 4 * c);
        float2& u = f.A[OF::ap(s, 2 * c)];
        float2& w = f.A[OF::ap(s, 2 * c + 1)];
        u = __fadd2_rn(__fadd2_rn(u, __fadd2_rn(two(-ea0), make_float2(q.x, q.y))), two(-nug));
        w = __fadd2_rn(__fadd2_rn(w, __fadd2_rn(two(-ea0), make_float2(q.z, q.w))), two(-nug));
      }
      const float en = ea0 + nug;
      set_diag(Sc, -2.0f * en);
      if (s > 0 || r) f.A[OF::ap(s, 0)].x = en;  // column 0
      yv[s] = ((ea0 + e0i) - yv[s]) + nug;
    });
    if (r == 0) {  // row 0
      f.A[0].x = -k0;
      yv[0] = -(e0i + nug);
    }
  } else {
    static_for<0, R>([&](auto Sc) {
      set_diag(Sc, -k0);
      yv[decltype(Sc)::value] = -yv[decltype(Sc)::value];
    });
  }
  static_for<0, R>([&](auto Sc) {  // rows past k: identity padding
    constexpr int s = decltype(Sc)::value;
    if (8 * s + 7 >= k) {
      if (8 * s + r >= k) {
#pragma unroll
        for (int c = 0; c < 4 * (s + 1); c++) f.A[OF::ap(s, c)] = two(0.0f);
        set_diag(Sc, -1.0f);
        yv[s] = 0.0f;
      }
    }
  });
  __syncwarp();  // gamma_a0 is read
  DF s2{f.varw, 0.0f};
  bool clamped = false;
  float max_ratio = 1.0f;
  const float pfloor = fmaxf(kPdFloor * k0, kPivotMin);
#pragma unroll
  for (int s = 0; s < R; s++) f.b[s] = 0.0f;
  static_for<0, K>([&](auto Jc) {
    constexpr int j = decltype(Jc)::value;
    constexpr int sj = j / 8, rj = j % 8, cj = j / 2;  // column pair of j
    float2 Lj[(j + 3) / 4 * 2 + 2];
#pragma unroll
    for (int c = 0; c < (j + 3) / 4; c++) {
      const float4 q = *reinterpret_cast<const float4*>(S + OL::row_off(j) + 4 * c);
      Lj[2 * c] = make_float2(q.x, q.y);
      Lj[2 * c + 1] = make_float2(q.z, q.w);
    }
    float nt[R];  // -(M_aj - sum_m L_am L_jm) of the lane's rows
    static_for<sj, R>([&](auto Sc) {
      constexpr int s = decltype(Sc)::value;
      const float2 m0 = f.A[OF::ap(s, cj)];
      float2 acc = make_float2(j & 1 ? m0.y : m0.x, 0.0f);
#pragma unroll
      for (int c = 0; c < j / 4 * 2; c++) acc = __ffma2_rn(f.A[OF::ap(s, c)], Lj[c], acc);
#pragma unroll
      for (int m = j / 4 * 4; m < j; m++)
        acc.x = m & 1 ? __fmaf_rn(f.A[OF::ap(s, m / 2)].y, Lj[m / 2].y, acc.x)
                      : __fmaf_rn(f.A[OF::ap(s, m / 2)].x, Lj[m / 2].x, acc.x);
      nt[s] = acc.x + acc.y;
    });
    float piv = -__shfl_sync(full, nt[sj], rj, 8);
    if (!(piv > pfloor)) {
      piv = pfloor;
      clamped = true;
    }
    const float inv = rcp_newton(sqrt_newton(piv));
    const float2 mj = f.A[OF::ap(sj, cj)];
    if (r == rj) max_ratio = fmaxf(max_ratio, -(j & 1 ? mj.y : mj.x) * inv * inv);
    const float yj = __shfl_sync(full, yv[sj], rj, 8) * inv;
    s2 = df_sub_square(s2, yj);
    if (r == rj) f.b[sj] = yj;
    static_for<sj, R>([&](auto Sc) {  // rows up to j: not used any more
      constexpr int s = decltype(Sc)::value;
      const float l = nt[s] * -inv;
      if (j & 1) f.A[OF::ap(s, cj)].y = l; else f.A[OF::ap(s, cj)].x = l;
      yv[s] = __fmaf_rn(l, -yj, yv[s]);
    });
    S[OL::row_off(j) + j] = inv;
    if constexpr (j + 1 < K) {  // row j + 1 is complete
      constexpr int sn = (j + 1) / 8;
      if (r == (j + 1) % 8) {
#pragma unroll
        for (int c = 0; c < j / 4 + 1; c++) {
          const float2 u = f.A[OF::ap(sn, 2 * c)], w = f.A[OF::ap(sn, 2 * c + 1)];
          *reinterpret_cast<float4*>(S + OL::row_off(j + 1) + 4 * c) =
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
#pragma unroll
  for (int o = 4; o; o >>= 1) max_ratio = fmaxf(max_ratio, __shfl_xor_sync(full, max_ratio, o));
  f.max_ratio = max_ratio;
  f.sigma = sqrtf(sig2);
  __syncwarp();
  oct_back_solve<K>(S, r, f.b);
  // increment form: b_0 = 1 + beta_0 - sum_{a>=1} beta_a (padding entries are zero)
  const float sb = oct_sum_from_1<K>(f.b);
  if (inc && r == 0) f.b[0] = (1.0f + f.b[0]) - sb;
  // a non-finite weight makes the sum so
  f.finite = isfinite(sb) && isfinite(__shfl_sync(full, f.b[0], 0, 8));
}

template <int K>
__device__ __forceinline__ bool oct_needs_rescue(const OctFactor<K>& f, const KernF& kf) {
  return f.clamped || row_error_too_large(f.max_ratio, f.varw, f.sigma, kf) || !isfinite(f.sigma) ||
         !f.finite;
}

// The field at the neighbours of the lane's slots (zero past k).
template <int K, bool LEVEL>
__device__ __forceinline__ void oct_gather(float (&vv)[K / 8], int r, int k,
                                           const int32_t* __restrict__ row, const float* v,
                                           uint64_t pol) {
#pragma unroll
  for (int s = 0; s < K / 8; s++) {
    vv[s] = 0.0f;
    if (8 * s + r < k) {
      const float* p = v + __ldg(row + 8 * s + r);
      vv[s] = LEVEL ? ld_level_f(p, pol) : ld_keep_f(p, pol);
    }
  }
}

// sum_a b_a v[c_a] in the stored sweeps' summation order (sweepsync.cuh), on
// every lane: slice h of the kp entries on lane h, from shared memory.
template <int K>
__device__ __forceinline__ float oct_dot(const float (&b)[K / 8], const float (&vv)[K / 8],
                                         float* S, int r, int kp) {
  using OL = OctLayout<K>;
  __syncwarp();
#pragma unroll
  for (int s = 0; s < K / 8; s++) {
    S[OL::kVecB + 8 * s + r] = b[s];
    S[OL::kVecV + 8 * s + r] = vv[s];
  }
  __syncwarp();
  const int lanes = gen_lanes(kp), hp = kp / lanes;
  float acc0 = 0.0f, acc1 = 0.0f;
  if (r < lanes) {
    const float4* bp = reinterpret_cast<const float4*>(S + OL::kVecB + r * hp);
    const float4* vp = reinterpret_cast<const float4*>(S + OL::kVecV + r * hp);
    for (int q = 0; q < hp / 4; q++) {
      const float4 w = bp[q], x = vp[q];
      acc0 = fmaf(w.x, x.x, acc0);
      acc1 = fmaf(w.y, x.y, acc1);
      acc0 = fmaf(w.z, x.z, acc0);
      acc1 = fmaf(w.w, x.w, acc1);
    }
  }
  float acc = acc0 + acc1;
  if (lanes >= 4) acc += __shfl_xor_sync(0xffffffffu, acc, 2, 8);
  if (lanes >= 2) acc += __shfl_xor_sync(0xffffffffu, acc, 1, 8);
  return __shfl_sync(0xffffffffu, acc, 0, 8);
}

// The FP64 conditional of a row out of line: the rescue is rare, and inlined its
// state would raise the register count of the whole kernel.
template <int K, int KT>
__device__ __noinline__ WarpRow64 oct_row64(const float4* __restrict__ xs, const int32_t* row,
                                            int k, float4 xq, KernF kf, double* W) {
  return warp_row_factor64<K, KT>(xs, row, k, xq, kf, W);
}

// The rows of the warp's points with `need` set recomputed in FP64, one at a
// time by the whole warp (warp_row_factor64); the lanes of such a point receive
// their weights, sigma and floor flag.  A collective; Sw: the shared memory of
// the warp's points, which is overwritten.
template <int K, int KT>
__device__ __forceinline__ void oct_rescue(OctFactor<K>& f, bool need, float* Sw, int r,
                                           const float4* __restrict__ xs, const int32_t* row, int k,
                                           float4 xq, const KernF& kf) {
  static_assert(4 * OctLayout<K>::kStride * sizeof(float) >= K * (K + 1) * sizeof(double), "");
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  unsigned m = __ballot_sync(full, need) & 0x01010101u;
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
    const WarpRow64 w = oct_row64<K, KT>(xs, rw, k, q, kf, reinterpret_cast<double*>(Sw));
    const float b = lane < k ? (float)w.b : 0.0f;
#pragma unroll
    for (int s = 0; s < K / 8; s++) {
      const float bs = __shfl_sync(full, b, 8 * s + r);
      if ((lane & ~7) == src) f.b[s] = bs;
    }
    if ((lane & ~7) == src) {
      f.sigma = (float)w.sigma;
      f.clamped = w.clamped;
    }
    __syncwarp();
  }
}

// The per-row factor backward after oct_factor: g = K_cc^-1 (alpha v_c), then row
// a of Kbar_cc, -g_a b_c + sbar b_a b_c over all c, and (a, i) against
// dkappa/dtheta, in FP32 in the order of the columns; the rows' sums meet in a
// fixed tree.  As in pair_row_backward the order is kept because the terms
// cancel; a lane therefore evaluates the values of its rows on both sides of
// the diagonal (taking each pair once saved 2 ms of the 12.1 above and was up
// to 1e-5 of the gradient apart).  Every lane of the warp must call this; `act`
// says whether the point counts.  The vectors of S are overwritten.
template <int K, int KT>
__device__ __forceinline__ void oct_row_backward(const OctFactor<K>& f, float* S, int r, int k,
                                                 const KernF& kf, float4 xq,
                                                 const float (&vv)[K / 8], float alpha, float sbar,
                                                 bool act, double& tl, double& ts, double& tn) {
  using OL = OctLayout<K>;
  using OF = OctFactor<K>;
  constexpr int R = K / 8;
  const unsigned full = 0xffffffffu;
  const float inv_s2 = 1.0f / kf.s2;
  float g[R], z[R];
#pragma unroll
  for (int s = 0; s < R; s++) g[s] = 8 * s + r < k ? alpha * vv[s] : 0.0f;
  const float r0 = __shfl_sync(full, g[0], 0, 8);
  if (f.inc) {
#pragma unroll
    for (int s = 0; s < R; s++)
      if (8 * s + r >= 1 && 8 * s + r < k) g[s] -= r0;
  }
  static_for<0, K>([&](auto Jc) {
    constexpr int j = decltype(Jc)::value;
    constexpr int sj = j / 8, rj = j % 8, cj = j / 2;
    const float zj = __shfl_sync(full, g[sj], rj, 8) * S[OL::row_off(j) + j];
    if (r == rj) z[sj] = zj;
    static_for<sj, R>([&](auto Sc) {  // rows up to j: not used any more
      constexpr int s = decltype(Sc)::value;
      const float2 l = f.A[OF::ap(s, cj)];
      g[s] = __fmaf_rn(j & 1 ? l.y : l.x, -zj, g[s]);
    });
  });
  oct_back_solve<K>(S, r, z);
  const float sg = oct_sum_from_1<K>(z);
  if (f.inc && r == 0) z[0] -= sg;
  const float* B = S + OL::kVecB;
  __syncwarp();
#pragma unroll
  for (int s = 0; s < R; s++) S[OL::kVecB + 8 * s + r] = f.b[s];
  __syncwarp();
  RowTheta th[R];
  float pn[R];
#pragma unroll
  for (int s = 0; s < R; s++) {
    const int a = 8 * s + r;
    const float ax = S[a], ay = S[K + a], az = S[2 * K + a];
    const float ba = f.b[s], sba = __fmul_rn(sbar, ba), ga = z[s];
    th[s] = RowTheta{0.0f, 0.0f};
    pn[s] = 0.0f;
    if (8 * s >= k) continue;  // the same on every lane
#pragma unroll 1
    for (int c = 0; c < k; c += 4) {
      const float4 X = *reinterpret_cast<const float4*>(S + c);
      const float4 Y = *reinterpret_cast<const float4*>(S + K + c);
      const float4 Z = *reinterpret_cast<const float4*>(S + 2 * K + c);
      const float4 Bc = *reinterpret_cast<const float4*>(B + c);
      const DPair d0 = dentry_pair<KT>(
          kf, sqdist2(sub2(ax, make_float2(X.x, X.y)), sub2(ay, make_float2(Y.x, Y.y)),
                      sub2(az, make_float2(Z.x, Z.y))));
      const DPair d1 = dentry_pair<KT>(
          kf, sqdist2(sub2(ax, make_float2(X.z, X.w)), sub2(ay, make_float2(Y.z, Y.w)),
                      sub2(az, make_float2(Z.z, Z.w))));
      auto term = [&](float bc, float kv, float lv, int cc) {
        const float kb = __fmaf_rn(sba, bc, __fmul_rn(-ga, bc));
        if (cc == a) {
          th[s].s += kb;
          pn[s] = kb;
        } else if (cc < k) {
          th[s].add(kb, kv, lv, inv_s2);
        }
      };
      term(Bc.x, d0.k.x, d0.l.x, c);
      term(Bc.y, d0.k.y, d0.l.y, c + 1);
      term(Bc.z, d1.k.x, d1.l.x, c + 2);
      term(Bc.w, d1.k.y, d1.l.y, c + 3);
    }
    const DPair dq =
        dentry_pair<KT>(kf, sqdist2(two(ax - xq.x), two(ay - xq.y), two(az - xq.z)));
    th[s].add(__fmaf_rn(-2.0f * sbar, ba, ga), dq.k.x, dq.l.x, inv_s2);
    if (a >= k) {
      th[s] = RowTheta{0.0f, 0.0f};
      pn[s] = 0.0f;
    }
  }
  if (r == 0) {  // Kbar_ii = sbar, on row 0
    th[0].s += sbar;
    pn[0] += sbar;
  }
  // sum over 32 rows: 16 apart, then 8, 4, 2, 1
  auto total = [&](auto get) {
    float x = R == 4 ? (get(0) + get(2)) + (get(1) + get(3 % R)) : (get(0) + get(2)) + get(1);
#pragma unroll
    for (int o = 4; o; o >>= 1) x += __shfl_xor_sync(full, x, o, 8);
    return x;
  };
  const float pl = total([&](int s) { return th[s].l; });
  const float ps = total([&](int s) { return th[s].s; });
  const float pnn = total([&](int s) { return pn[s]; });
  if (act && r == 0) {
    tl += pl;
    ts += ps;
    tn += pnn;
  }
}

}  // namespace ggp
