// Adjoints (Sec. 2.3: forward and backward derivatives of the conditioning
// steps, differentiated through the Cholesky factor).
//
// With every sparse row written as v_i = b_i . v_c(i) + sigma_i xi_i:
//  * whiten VJP (xi = L^-1 v, cotangent xibar, logdetbar), w_i = xibar_i/sigma_i:
//      vbar_i = w_i - sum over children (j, a) of i of w_j b_ja   (every row
//      j scatters -w_j b_ja to its neighbours), bbar_i = -w_i v_c, sigbar_i =
//      -w_i xi_i + 2 logdetbar / sigma_i;
//  * generate VJP (v = L xi, cotangent vbar): u = (I - B)^-T vbar by a reverse
//      level sweep, u_j = vbar_j + sum over children (i, a) of j of b_ia u_i
//      (every row i, once u_i is complete, scatters b_ia u_i to its
//      neighbours); xibar_i = sigma_i u_i, bbar_i = u_i v_c, sigbar_i = u_i xi_i;
//  * factor backward, per row, from b = K_cc^-1 K_ci and s = sigma^2:
//      sbar = sigbar/(2 sigma), g = K_cc^-1 bbar, Kbar_cc = -g b^T + sbar b b^T,
//      Kbar_ci = g - 2 sbar b, Kbar_ii = sbar, theta_bar += sum Kbar dK/dtheta.
//    The factors are recomputed (bit-identical to the forward), not stored.
//  * dense block (L0 = chol(K_00)): Lbar0 from the sweep, then
//      Kbar_00 = L0^-T Phi(L0^T Lbar0) L0^-1 (Phi: lower triangle, halved
//      diagonal), theta_bar += sum Kbar_00 dK_00/dtheta.
//  * NLL value and gradient in one pass (graphgp_nll_grad_fused): per row the
//      factor, xi_i, the value's terms, the whiten-VJP scatter and the
//      factor backward above, each conditional computed once.
// theta = (lengthscale, sigma2, nugget); theta_bar is accumulated in FP64.
#include <algorithm>

#include "pointoct.cuh"
#include "pointwide.cuh"

namespace ggp {
namespace {

// ---- dense helpers ------------------------------------------------------------
// y_m (+)= sum_{i >= m} M[i][m] x_i (transpose of a lower-triangular n0 x n0 M).
// A block takes 32 columns: its warps stage kTmvRows rows of them at once, then
// one warp adds down the columns, so that the sum keeps its order (ascending i,
// one accumulator).  Bound by that chain and two memory latencies per chunk; a
// thread per column waited for one load after another: n0 = 256
// 66 -> 5.3 us.
constexpr int kTmvRows = 256;

template <bool ACC>
__global__ void __launch_bounds__(256) dense_lower_tmatvec_kernel(
    const float* __restrict__ M, const float* __restrict__ x, float* __restrict__ y, int n0) {
  __shared__ float s_m[kTmvRows][32], s_x[kTmvRows];
  const int c = threadIdx.x & 31, w = threadIdx.x >> 5, m0 = blockIdx.x * 32, m = m0 + c;
  float s = 0.0f;
  for (int i0 = m0; i0 < n0; i0 += kTmvRows) {
    const int rows = min(kTmvRows, n0 - i0);
    float r[kTmvRows / 8];
#pragma unroll
    for (int t = 0; t < kTmvRows / 8; t++) {
      const int i = i0 + w + 8 * t;
      r[t] = (i < n0 && m < n0) ? M[(int64_t)i * n0 + m] : 0.0f;
    }
    const float xr = (int)threadIdx.x < rows ? x[i0 + threadIdx.x] : 0.0f;
    __syncthreads();  // the chunk before has been read
#pragma unroll
    for (int t = 0; t < kTmvRows / 8; t++) s_m[w + 8 * t][c] = r[t];
    s_x[threadIdx.x] = xr;
    __syncthreads();
    if (w == 0) {
#pragma unroll 16
      for (int t = 0; t < rows; t++)
        if (i0 + t >= m) s = fmaf(s_m[t][c], s_x[t], s);
    }
  }
  if (w == 0 && m < n0) y[m] = ACC ? y[m] + s : s;
}

// Lbar0[a][b] = sgn * u_a xi_b (b <= a) plus diag 2 logdetbar / L0_aa.
__global__ void dense_lbar_kernel(const float* __restrict__ u, const float* __restrict__ xi,
                                  const float* __restrict__ L0, int n0, float sgn, float ldbar,
                                  float* __restrict__ out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)n0 * n0;
       e += (int64_t)gridDim.x * blockDim.x) {
    int a = (int)(e / n0), b = (int)(e % n0);
    float v = 0.0f;
    if (b <= a) v = sgn * u[a] * xi[b];
    if (a == b) v += 2.0f * ldbar / L0[e];
    out[e] = v;
  }
}

// C = op(A) B for n x n row-major matrices; op(A) = A^T when TRANS.  If PHI,
// keeps the lower triangle of the result with the diagonal halved.  32 x 32 of C
// per block from 32-row chunks of both operands in shared memory, the next chunk
// loaded meanwhile; a thread has four neighbouring entries, each one accumulator
// over ascending m.  At n = 256 there are 64 tiles, so a chunk's latency bounds
// it; a thread per entry that read both operands from L2
// took 34 us (n = 256), this 10-13 us.
constexpr int kGemmTile = 32;

template <bool TRANS, bool PHI>
__global__ void __launch_bounds__(256) dense_gemm_kernel(const float* __restrict__ A,
                                                         const float* __restrict__ B,
                                                         float* __restrict__ C, int n) {
  constexpr int T = kGemmTile;
  __shared__ float s_a[T][T + 1];              // [m][row of C]
  __shared__ __align__(16) float s_b[T][T];    // [m][column of C]
  const int a0 = blockIdx.y * T, b0 = blockIdx.x * T;
  const int lx = threadIdx.x & 31, ly = threadIdx.x >> 5;  // loads: 8 rows of 32
  const int row = threadIdx.x >> 3, col = (threadIdx.x & 7) * 4;
  float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  if (!PHI || b0 <= a0) {
    float ra[4], rb[4];
    auto load = [&](int m0) {
#pragma unroll
      for (int t = 0; t < 4; t++) {
        const int y = ly + 8 * t, m = m0 + y;
        if (TRANS)
          ra[t] = (m < n && a0 + lx < n) ? A[(int64_t)m * n + a0 + lx] : 0.0f;
        else
          ra[t] = (a0 + y < n && m0 + lx < n) ? A[(int64_t)(a0 + y) * n + m0 + lx] : 0.0f;
        rb[t] = (m < n && b0 + lx < n) ? B[(int64_t)m * n + b0 + lx] : 0.0f;
      }
    };
    load(0);
    for (int m0 = 0; m0 < n; m0 += T) {
      __syncthreads();  // the chunk before has been read
#pragma unroll
      for (int t = 0; t < 4; t++) {
        const int y = ly + 8 * t;
        if (TRANS)
          s_a[y][lx] = ra[t];
        else
          s_a[lx][y] = ra[t];
        s_b[y][lx] = rb[t];
      }
      __syncthreads();
      if (m0 + T < n) load(m0 + T);
#pragma unroll
      for (int m = 0; m < T; m++) {
        const float a = s_a[m][row];
        const float4 v = *reinterpret_cast<const float4*>(&s_b[m][col]);
        s[0] = fmaf(a, v.x, s[0]);
        s[1] = fmaf(a, v.y, s[1]);
        s[2] = fmaf(a, v.z, s[2]);
        s[3] = fmaf(a, v.w, s[3]);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < 4; q++) {
    const int a = a0 + row, b = b0 + col + q;
    if (a < n && b < n) {
      float out = s[q];
      if (PHI) out = b > a ? 0.0f : (a == b ? 0.5f * out : out);
      C[(int64_t)a * n + b] = out;
    }
  }
}

__device__ void block_add3(double t0, double t1, double t2, double* out) {
  __shared__ double red[3][32];
  for (int o = 16; o; o >>= 1) {
    t0 += __shfl_xor_sync(0xffffffffu, t0, o);
    t1 += __shfl_xor_sync(0xffffffffu, t1, o);
    t2 += __shfl_xor_sync(0xffffffffu, t2, o);
  }
  int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    red[0][w] = t0;
    red[1][w] = t1;
    red[2][w] = t2;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double s0 = 0, s1 = 0, s2 = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); i++) {
      s0 += red[0][i];
      s1 += red[1][i];
      s2 += red[2][i];
    }
    atomicAdd(out + 0, s0);
    atomicAdd(out + 1, s1);
    atomicAdd(out + 2, s2);
  }
  __syncthreads();  // the partials may be reused by a following call
}

// theta_bar += sum_{a,b} Kbar[a][b] dK_ab/dtheta over the dense block.
template <int KT>
__global__ void dense_theta_kernel(const float* __restrict__ Kbar, const float4* __restrict__ xs,
                                   int n0, KernF kf, double unit, double* __restrict__ thetabar) {
  double tl = 0, ts = 0, tn = 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)n0 * n0;
       e += (int64_t)gridDim.x * blockDim.x) {
    int a = (int)(e / n0), b = (int)(e % n0);
    float kb = Kbar[e];
    if (a == b) {
      ts += kb;
      tn += kb;
    } else {
      float d2 = sqdist(xs[a], xs[b]);
      ts += (double)(kb * kappa_d2<KT>(kf, d2) / kf.s2);
      tl += (double)(kb * dkappa_dell_d2<KT>(kf, d2));
    }
  }
  block_add3(tl * unit, ts, tn, thetabar);
}

// ---- adjoint sweeps by scatter ------------------------------------------------
// Both VJPs apply a transpose of the row operator: entry b_ia of row i moves
// a cotangent from position i to its neighbour c_a.  Rows are streamed in
// position order, LANES threads per row as in the forward sweeps (16-byte
// row loads), and each entry's contribution is added at its neighbour with a
// fire-and-forget atomic add in L2 (red.global.add.f32).  The additions into
// one position arrive in no fixed order, so results agree with the ordered
// sums to rounding, not bit for bit.
#define GGP_ADJ_KP_DISPATCH(kp, call) \
  switch (kp) {                       \
    case 4: call(4); break;           \
    case 8: call(8); break;           \
    case 12: call(12); break;         \
    case 16: call(16); break;         \
    case 20: call(20); break;         \
    case 24: call(24); break;         \
    case 28: call(28); break;         \
    case 32: call(32); break;         \
    case 48: call(48); break;         \
    default: call(64); break;         \
  }

template <int HP>
__device__ __forceinline__ void load_row_slice(int4 (&n)[HP / 4], float4 (&w)[HP / 4],
                                               const int32_t* __restrict__ nbr,
                                               const float* __restrict__ b, int64_t off,
                                               uint64_t pol) {
#pragma unroll
  for (int c = 0; c < HP / 4; c++) {
    n[c] = ld_stream_i4(reinterpret_cast<const int4*>(nbr + off) + c, pol);
    w[c] = ld_stream_f4(reinterpret_cast<const float4*>(b + off) + c, pol);
  }
}

template <int HP>
__device__ __forceinline__ void scatter_row(float* y, const int4 (&n)[HP / 4],
                                            const float4 (&w)[HP / 4], float a) {
  // padded entries (weight 0, neighbour 0) add nothing and are skipped
#pragma unroll
  for (int c = 0; c < HP / 4; c++) {
    if (w[c].x != 0.0f) atomicAdd(y + n[c].x, w[c].x * a);
    if (w[c].y != 0.0f) atomicAdd(y + n[c].y, w[c].y * a);
    if (w[c].z != 0.0f) atomicAdd(y + n[c].z, w[c].z * a);
    if (w[c].w != 0.0f) atomicAdd(y + n[c].w, w[c].w * a);
  }
}

// whiten VJP, sparse rows at positions [p_begin, p_end): vbar_p += w_p and
// vbar_c -= w_j b_j,c for every row j, w_j = xibar_j / sigma_j (for the whole
// graph vbar's sparse entries start at 0, its dense entries at
// L0^-T xibar_0).  No ordering between rows.
template <int KP>
__global__ void __launch_bounds__(256) whiten_adjoint_scatter_kernel(
    const int32_t* __restrict__ nbr, const float* __restrict__ b, const float* __restrict__ sigma,
    const float* __restrict__ xibar, float* vbar, int64_t n0, int64_t p_begin, int64_t p_end) {
  constexpr int LANES = gen_lanes(KP), HP = KP / LANES, GPB = 256 / LANES;
  const int h = threadIdx.x % LANES;
  const uint64_t pol = l2_evict_first();
  const int64_t stride = (int64_t)gridDim.x * GPB;
  for (int64_t p = p_begin + (int64_t)blockIdx.x * GPB + threadIdx.x / LANES; p < p_end;
       p += stride) {
    int4 n[HP / 4];
    float4 w[HP / 4];
    load_row_slice<HP>(n, w, nbr, b, (p - n0) * KP + h * HP, pol);
    const float a = xibar[p] / sigma[p];
    if (h == 0) atomicAdd(vbar + p, a);
    scatter_row<HP>(vbar, n, w, -a);
  }
}

// generate VJP: u = (I - B)^-T vbar.  u starts as vbar; deepest level first,
// every row i of level l -- whose u_i is complete, all its children lying in
// deeper levels -- adds b_ia u_i at each neighbour c_a.  One cooperative
// launch, a grid-wide barrier between levels (the barrier's release orders a
// block's atomics before the next level's reads); the first row of a block's
// slice is loaded before the wait.
template <int KP>
__global__ void __launch_bounds__(256) generate_adjoint_scatter_kernel(
    const int32_t* __restrict__ nbr, const float* __restrict__ b, float* u,
    const int64_t* __restrict__ level_off, int l_first, int num_levels, int64_t n0,
    LevelBarrier lb) {
  constexpr int LANES = gen_lanes(KP), HP = KP / LANES, GPB = 256 / LANES;
  __shared__ int s_flag;
  const int h = threadIdx.x % LANES;
  const uint64_t pol = l2_evict_first();
  const uint64_t pol_u = l2_evict_last();
  for (int l = num_levels - 1; l >= l_first; l--) {
    const int64_t lo = level_off[l], cnt = level_off[l + 1] - lo;
    const int64_t per = (cnt + gridDim.x - 1) / gridDim.x;
    const int64_t b0 = lo + min((int64_t)blockIdx.x * per, cnt);
    const int64_t hi = lo + min((int64_t)(blockIdx.x + 1) * per, cnt);
    int64_t p = b0 + threadIdx.x / LANES;
    int4 n[HP / 4];
    float4 w[HP / 4];
    if (p < hi) load_row_slice<HP>(n, w, nbr, b, (p - n0) * KP + h * HP, pol);
    if (l < num_levels - 1 && lb.wait(l + 1, gridDim.x, &s_flag)) return;
    while (p < hi) {
      const float a = ld_coherent_f(u + p, pol_u);
      int4 nn[HP / 4];
      float4 ww[HP / 4];
#pragma unroll
      for (int c = 0; c < HP / 4; c++) {
        nn[c] = n[c];
        ww[c] = w[c];
      }
      p += GPB;
      if (p < hi) load_row_slice<HP>(n, w, nbr, b, (p - n0) * KP + h * HP, pol);
      scatter_row<HP>(u, nn, ww, a);
    }
    __syncthreads();
    lb.arrive(l);
  }
}

// generate VJP, the levels the sweep ends with (the first of the graph, a few
// dozen points each): one block with u up to their end in shared memory, so a
// level costs a block barrier and shared-memory atomics instead of a grid barrier
// and a round trip through L2.  Rows are loaded D steps ahead, across levels.
// Bound by the shared-memory atomics, so the run ends at the first level with
// more than kHeadEntries row entries.  The vector-only VJP with no such run / one
// up to 64 / 128 / 256 / 512 points a level, us: 127001 points, k = 16: 221 / 200 /
// 192 / 192 / 202; k = 48: 713 / 653 / 641 / 674 / 800; k = 7 (padded to 8): 123 /
// 126 / 122 / 118 / 118; 10^6, k = 16: 427 / 408 / 390 / 382 / 386.
constexpr int kHeadThreads = 512;
constexpr int64_t kHeadPoints = 49152;  // positions held (192 KB)
constexpr int kHeadLevels = 4096;
constexpr int64_t kHeadEntries = 4096;  // row entries of its largest level

template <int KP>
__global__ void __launch_bounds__(kHeadThreads, 1) generate_adjoint_head_kernel(
    const int32_t* __restrict__ nbr, const float* __restrict__ b, float* __restrict__ u,
    const int64_t* __restrict__ level_off, int l_end, int64_t n0) {
  constexpr int LANES = gen_lanes(KP), HP = KP / LANES, PPB = kHeadThreads / LANES;
  constexpr int D = HP <= 4 ? 3 : (HP <= 8 ? 2 : 1);
  extern __shared__ float s_u[];  // u up to the last level's end, then the offsets
  const int32_t end = (int32_t)level_off[l_end];
  int32_t* s_lo = reinterpret_cast<int32_t*>(s_u + end);
  for (int l = threadIdx.x; l <= l_end; l += kHeadThreads) s_lo[l] = (int32_t)level_off[l];
  for (int i = threadIdx.x; i < end; i += kHeadThreads) s_u[i] = u[i];
  __syncthreads();
  const int h = threadIdx.x % LANES, slot = threadIdx.x / LANES;
  const uint64_t pol = l2_policy<0>();
  int4 n[D + 1][HP / 4];
  float4 w[D + 1][HP / 4];
  int ll = l_end - 1, lp = s_lo[ll];  // the next step to load
  auto load = [&](int4 (&nn)[HP / 4], float4 (&ww)[HP / 4]) {
    if (ll < 1) return;
    const int q = lp + slot;
    if (q < s_lo[ll + 1]) load_row_slice<HP>(nn, ww, nbr, b, ((int64_t)q - n0) * KP + h * HP, pol);
    lp += PPB;
    if (lp >= s_lo[ll + 1]) lp = s_lo[--ll];
  };
#pragma unroll
  for (int i = 0; i < D; i++) load(n[i], w[i]);
  int l = l_end - 1, p = s_lo[l];
  while (l >= 1) {
#pragma unroll
    for (int i = 0; i <= D; i++) {  // buffer i holds this step, i + D is refilled
      if (l < 1) break;
      load(n[(i + D) % (D + 1)], w[(i + D) % (D + 1)]);
      if (p == s_lo[l]) __syncthreads();  // the levels behind are complete
      const int q = p + slot;
      if (q < s_lo[l + 1]) scatter_row<HP>(s_u, n[i], w[i], s_u[q]);
      p += PPB;
      if (p >= s_lo[l + 1]) p = s_lo[--l];
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < end; i += kHeadThreads) u[i] = s_u[i];
}

int whiten_adjoint_scatter(graphgp_graph_t g, graphgp_factor_t f, const float* xibar, float* vbar,
                           int64_t p_begin, int64_t p_end, cudaStream_t s) {
  const int64_t grid = std::min<int64_t>((p_end - p_begin + 63) / 64, (int64_t)num_sms() * 8);
#define GGP_WSC(KP)                                                                              \
  whiten_adjoint_scatter_kernel<KP><<<(unsigned)grid, 256, 0, s>>>(g->nbr, f->b, f->sigma, xibar, \
                                                                   vbar, g->n0, p_begin, p_end)
  GGP_ADJ_KP_DISPATCH(g->kp, GGP_WSC);
#undef GGP_WSC
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

// ---- per-row factor backward ------------------------------------------------------
// mode 0 (whiten): alpha_i = -xibar_i / sigma_i, beta = 2 logdetbar.
// mode 1 (generate): alpha_i = u_i, beta = 0; also writes xibar_i = sigma_i u_i.
// bbar_i = alpha_i v_c(i), sigbar_i = alpha_i xi_i + beta / sigma_i.
// 16 < k <= 32: eight lanes per point, the factor recomputed by oct_factor
// (bit-identical b and sigma to the forward kernel).  Rows the forward factor
// recomputed in FP64 (rescue.cuh) go to factor_backward_rescue_kernel, whose
// list holds every row.
template <int K, int KT>
__global__ void __launch_bounds__(kPairThreads, OctLayout<K>::kBlocks) factor_backward_oct_kernel(
    const float4* __restrict__ xs, const int32_t* __restrict__ nbr, int64_t N, int k, int kp,
    int64_t n0, KernF kf, double unit, int mode, const float* __restrict__ coef, float beta,
    const float* __restrict__ v, const float* __restrict__ xi, float* __restrict__ xibar_out,
    double* __restrict__ thetabar, int64_t* __restrict__ rescue_rows,
    unsigned long long* __restrict__ rescue_count) {
  using OL = OctLayout<K>;
  extern __shared__ __align__(16) float psm[];
  const int lane = threadIdx.x & 31, r = lane & 7, first = (threadIdx.x >> 5) * 4;
  float* S = psm + (threadIdx.x >> 3) * OL::kStride;
  const uint64_t pol_v = l2_evict_last();
  double tl = 0.0, ts = 0.0, tn = 0.0;
  const int64_t npts = N - n0;
  const int64_t stride = (int64_t)gridDim.x * OL::kPoints;
  for (int64_t b0 = (int64_t)blockIdx.x * OL::kPoints; b0 < npts; b0 += stride) {
    __syncthreads();  // the warps of a block share the instruction stream
    const int64_t t = b0 + first + (lane >> 3);
    const bool valid = t < npts;
    const int64_t tt = valid ? t : npts - 1, i = n0 + tt;
    const int32_t* row = nbr + tt * kp;
    const float4 xq = __ldg(xs + i);
    oct_stage<K>(S, r, xs, row, kp);
    OctFactor<K> f;
    oct_factor<K, KT>(f, S, r, k, kf, xq);
    const bool rescue = valid && oct_needs_rescue(f, kf);
    const float ci = coef[i], xii = xi[i];
    const float alpha = mode == 0 ? -ci / f.sigma : ci;
    const float sigbar = alpha * xii + beta / f.sigma;
    float vv[K / 8];
    oct_gather<K, false>(vv, r, k, row, v, pol_v);
    oct_row_backward<K, KT>(f, S, r, k, kf, xq, vv, alpha, sigbar / (2.0f * f.sigma),
                            valid && !rescue, tl, ts, tn);
    if (valid && r == 0) {
      if (rescue)
        rescue_rows[atomicAdd(rescue_count, 1ull)] = i;
      else if (mode == 1)
        xibar_out[i] = f.sigma * ci;
    }
  }
  block_add3(tl * unit, ts, tn, thetabar);
}

// The same per-row backward for 32 < k <= 64: one warp per point, the factor
// recomputed by point_factor_wide (bit-identical to the forward kernel), then
// g = K_cc^-1 bbar by two triangular solves in shared memory.  Lane a + 32 s
// takes row a + 32 s of Kbar against dK/dtheta (FP32 per row, FP64 across
// rows); rows needing the FP64 rescue go to factor_backward_rescue_kernel.
// Shared memory holds three blocks per SM, so the registers are set for three:
// left to itself the compiler takes 64 and shortens the unrolled loops (400,000
// rows, NLL gradient, k = 64: 52.6 ms with squared exponential, 56.3 Matern-3/2;
// 43.1 and 45.0 with three blocks).
template <int KT>
__global__ void __launch_bounds__(128, 3) factor_backward_wide_kernel(
    const float4* __restrict__ xs, const int32_t* __restrict__ nbr, int64_t N, int k, int kp,
    int64_t n0, KernF kf, double unit, int mode, const float* __restrict__ coef, float beta,
    const float* __restrict__ v, const float* __restrict__ xi, float* __restrict__ xibar_out,
    double* __restrict__ thetabar, int64_t* __restrict__ rescue_rows,
    unsigned long long* __restrict__ rescue_count) {
  extern __shared__ __align__(16) unsigned char wide_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  WideWarp& W = reinterpret_cast<WideWarp*>(wide_smem)[warp];
  double tl = 0.0, ts = 0.0, tn = 0.0;
  const float inv_s2 = 1.0f / kf.s2;
  const int64_t npts = N - n0;
  const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp; t < npts; t += nw) {
    const int64_t i = n0 + t;
    const int32_t* row = nbr + t * kp;
    for (int a = lane; a < k; a += 32) W.x[a] = __ldg(xs + row[a]);
    __syncwarp();
    const float4 xq = __ldg(xs + i);
    const WideFactor r = point_factor_wide<KT>(W, k, kf, xq);
    if (wide_needs_rescue(W, r, k, kf)) {
      if (lane == 0) rescue_rows[atomicAdd(rescue_count, 1ull)] = i;
      __syncwarp();
      continue;
    }
    const float sigma = r.sigma;
    const float ci = coef[i];
    const float alpha = mode == 0 ? -ci / sigma : ci;
    const float sigbar = alpha * xi[i] + beta / sigma;
    const float sbar = sigbar / (2.0f * sigma);
    for (int a = lane; a < k; a += 32) W.g[a] = alpha * v[row[a]];
    __syncwarp();
    wide_chol_solve(W, k, r.inc);
    for (int a = lane; a < k; a += 32) {
      const float ga = W.g[a], ba = W.y[a];
      const float4 xa = W.x[a];
      float pl = 0.0f, ps = 0.0f, pn = 0.0f;
      for (int c = 0; c < k; c++) {
        const float bc = W.y[c];
        const float kb = -ga * bc + sbar * ba * bc;
        if (c == a) {
          ps += kb;
          pn += kb;
        } else {
          const KD kd = kappa_dkappa_d2<KT>(kf, sqdist(xa, W.x[c]));
          ps += kb * kd.k * inv_s2;
          pl += kb * kd.dl;
        }
      }
      const float kci = ga - 2.0f * sbar * ba;
      const KD kq = kappa_dkappa_d2<KT>(kf, sqdist(xa, xq));
      ps += kci * kq.k * inv_s2;
      pl += kci * kq.dl;
      tl += pl;
      ts += ps;
      tn += pn;
    }
    if (lane == 0) {  // Kbar_ii = sbar
      ts += sbar;
      tn += sbar;
      if (mode == 1) xibar_out[i] = sigma * ci;
    }
    __syncwarp();
  }
  block_add3(tl * unit, ts, tn, thetabar);
}

// FP64 backward of the rows the per-row kernels handed over (rescue.cuh).
template <int G, int KT>
__global__ void __launch_bounds__(128) factor_backward_rescue_kernel(
    const float4* __restrict__ xs, const int32_t* __restrict__ nbr, int k, int kp, int64_t n0,
    KernF kf, double unit, int mode, const float* __restrict__ coef, float beta,
    const float* __restrict__ v, const float* __restrict__ xi, float* __restrict__ xibar_out,
    double* __restrict__ thetabar, const int64_t* __restrict__ rows,
    const unsigned long long* __restrict__ count, unsigned long long cap) {
  double tl = 0.0, ts = 0.0, tn = 0.0;
  const int64_t n = (int64_t)(*count < cap ? *count : cap);
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = rows[r];
    const int32_t* row_ptr = nbr + (i - n0) * kp;
    Row64<G> R;
    row_factor64<G, KT>(R, xs, row_ptr, k, xs[i], kf);
    const float sg = (float)R.sigma;
    const float ci = coef[i];
    const double al = mode == 0 ? -(double)ci / sg : (double)ci;
    const double sb = al * (double)xi[i] + (double)beta / sg;
    row_backward64<G, KT>(R, xs, row_ptr, k, xs[i], kf, v, al, sb, sg, tl, ts, tn);
    if (mode == 1) xibar_out[i] = sg * ci;
  }
  block_add3(tl * unit, ts, tn, thetabar);
}

// The per-row backward for k <= 16: two lanes per point, the factor recomputed
// by pair_factor (bit-identical b and sigma to the forward kernel).
template <int K, int KT>
__global__ void __launch_bounds__(kPairThreads, PairLayout<K>::kBlocks) factor_backward_pair_kernel(
    const float4* __restrict__ xs, const int32_t* __restrict__ nbr, int64_t N, int k, int64_t n0,
    KernF kf, double unit, int mode, const float* __restrict__ coef, float beta,
    const float* __restrict__ v, const float* __restrict__ xi, float* __restrict__ xibar_out,
    double* __restrict__ thetabar, int64_t* __restrict__ rescue_rows,
    unsigned long long* __restrict__ rescue_count, unsigned long long rescue_cap) {
  using PL = PairLayout<K>;
  extern __shared__ __align__(16) float psm[];
  const int lane = threadIdx.x & 31, r = lane & 1, first = (threadIdx.x >> 5) * 16;
  float* S = psm + (threadIdx.x >> 1) * PL::kStride;
  const uint64_t pol_v = l2_evict_last();
  double tl = 0.0, ts = 0.0, tn = 0.0;
  const int64_t npts = N - n0;
  const int64_t stride = (int64_t)gridDim.x * PL::kPoints;
  PairLoad<K> ld;
  for (int64_t b0 = (int64_t)blockIdx.x * PL::kPoints; b0 < npts; b0 += stride) {
    __syncthreads();  // the warps of a block share the instruction stream
    const int64_t t = b0 + first + (lane >> 1);
    const bool valid = t < npts;
    const int64_t tt = valid ? t : npts - 1, i = n0 + tt;
    const int32_t* row_ptr = nbr + tt * K;
    const float4 xq = __ldg(xs + i);
    ld.indices(r, row_ptr);
    ld.coords(r, xs);
    ld.stage(S, r);
    PairFactor<K> f;
    pair_factor<K, KT>(f, S, r, k, kf, xq);
    const bool rescue = valid && pair_needs_rescue(f, kf);
    const float ci = coef[i], xii = xi[i];
    const float alpha = mode == 0 ? -ci / f.sigma : ci;
    const float sigbar = alpha * xii + beta / f.sigma;
    float vv[K / 2];
    pair_gather<K, false>(vv, r, row_ptr, v, pol_v);
    pair_row_backward<K, KT>(f, S, r, k, kf, xq, vv, alpha, sigbar / (2.0f * f.sigma),
                             valid && !rescue, tl, ts, tn);
    if (valid && !rescue && r == 0 && mode == 1) xibar_out[i] = f.sigma * ci;
    if (rescue && r == 0) {
      // listed for factor_backward_rescue_kernel; recomputed here when the list is full
      const unsigned long long slot = atomicAdd(rescue_count, 1ull);
      if (slot < rescue_cap) {
        rescue_rows[slot] = i;
      } else {
        Row64<K> R;
        row_factor64<K, KT>(R, xs, row_ptr, k, xq, kf);
        const float sg = (float)R.sigma;
        const double al = mode == 0 ? -(double)ci / sg : (double)ci;
        const double sb = al * (double)xii + (double)beta / sg;
        row_backward64<K, KT>(R, xs, row_ptr, k, xq, kf, v, al, sb, sg, tl, ts, tn);
        if (mode == 1) xibar_out[i] = sg * ci;
      }
    }
    __syncwarp();
  }
  block_add3(tl * unit, ts, tn, thetabar);
}

// NLL value and gradient in one pass, the factors recomputed and never stored
// (k <= 16, two lanes per point).  Each row's b and sigma come from pair_factor
// with the factor kernel's FP64 rescue, so they are bit-identical to a stored
// factor's; xi_i = (v_i - b . v_c) / sigma_i follows the stored sweeps' order.
// The row then adds its share of what graphgp_nll + graphgp_nll_backward
// compute: xi_i^2 and log sigma_i to the value; w_i = nllbar xi_i / sigma_i at
// i and -w_i b_ia at each neighbour (vbar, atomic adds; vbar's sparse entries
// start at 0); and the row's factor backward with alpha = -w_i and sigbar =
// alpha xi_i + nllbar / sigma_i (the logdet cotangent nllbar / 2, doubled).
// Rows sent to FP64 follow the others of their warp, one at a time: they leave
// xi_i and nllbar xi_i in xi_out / xibar_out and are listed for
// factor_backward_rescue_kernel (recomputed here when the list is full).
template <int K, int KT>
__global__ void __launch_bounds__(kPairThreads, PairLayout<K>::kBlocks) nll_grad_fused_kernel(
    const float4* __restrict__ xs, const int32_t* __restrict__ nbr, int64_t N, int k, int64_t n0,
    KernF kf, double unit, float nllbar, const float* __restrict__ v, float* vbar,
    float* __restrict__ xi_out, float* __restrict__ xibar_out, double* __restrict__ thetabar,
    double* __restrict__ acc, unsigned long long* __restrict__ not_pd, int64_t* __restrict__ rescue_rows,
    unsigned long long* __restrict__ rescue_count, unsigned long long rescue_cap) {
  using PL = PairLayout<K>;
  extern __shared__ __align__(16) float psm[];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, r = lane & 1, first = (threadIdx.x >> 5) * 16;
  float* S = psm + (threadIdx.x >> 1) * PL::kStride;
  const uint64_t pol_v = l2_evict_last();
  LogAcc lacc;
  double sq = 0.0, tl = 0.0, ts = 0.0, tn = 0.0;
  unsigned long long clamped = 0;
  const int64_t npts = N - n0;
  const int64_t stride = (int64_t)gridDim.x * PL::kPoints;
  PairLoad<K> ld;
  for (int64_t b0 = (int64_t)blockIdx.x * PL::kPoints; b0 < npts; b0 += stride) {
    __syncthreads();  // the warps of a block share the instruction stream
    const int64_t t = b0 + first + (lane >> 1);
    const bool valid = t < npts;
    const int64_t tt = valid ? t : npts - 1, i = n0 + tt;
    const int32_t* row_ptr = nbr + tt * K;
    const float4 xq = __ldg(xs + i);
    ld.indices(r, row_ptr);
    ld.coords(r, xs);
    ld.stage(S, r);
    PairFactor<K> f;
    pair_factor<K, KT>(f, S, r, k, kf, xq);
    const bool rescue = valid && pair_needs_rescue(f, kf), act = valid && !rescue;
    float vv[K / 2];
    pair_gather<K, false>(vv, r, row_ptr, v, pol_v);
    const float sigma = f.sigma;
    const float xv = (ld_keep_f(v + i, pol_v) - pair_dot<K>(f.b, vv, r)) / sigma;
    const float xb = nllbar * xv;
    const float w = xb / sigma;
    if (act) {
      if (r == 0) {
        sq += (double)xv * (double)xv;
        lacc.mul(sigma);
        clamped += f.clamped ? 1 : 0;
        atomicAdd(vbar + i, w);
      }
#pragma unroll
      for (int s = 0; s < K / 2; s++) {
        const int2 c = __ldg(reinterpret_cast<const int2*>(row_ptr) + s);
        const float bs = pair_own<K>(f.b, r, s);
        if (bs != 0.0f) atomicAdd(vbar + (r ? c.y : c.x), bs * -w);
      }
    }
    const float alpha = -xb / sigma;
    const float sigbar = alpha * xv + nllbar / sigma;
    pair_row_backward<K, KT>(f, S, r, k, kf, xq, vv, alpha, sigbar / (2.0f * sigma), act, tl, ts,
                             tn);
    unsigned m = __ballot_sync(full, rescue && r == 0);
    while (m) {
      const int src = __ffs(m) - 1;
      m &= m - 1;
      __syncwarp();
      const int64_t u = b0 + first + (src >> 1), iu = n0 + u;
      const int32_t* row = nbr + u * K;
      const float4 xu = __ldg(xs + iu);
      const WarpRow64 wr = warp_row_factor64<K, KT>(
          xs, row, k, xu, kf, reinterpret_cast<double*>(psm + first * PL::kStride));
      const float b = lane < k ? (float)wr.b : 0.0f, sg = (float)wr.sigma;
      const float dot = warp_dot_stored_order<K>(b, row, v, pol_v);
      const float xu0 = __shfl_sync(full, (ld_keep_f(v + iu, pol_v) - dot) / sg, 0);
      const float xbu = nllbar * xu0, wu = xbu / sg;
      if (lane < k && b != 0.0f) atomicAdd(vbar + row[lane], b * -wu);
      if (lane == src) {
        sq += (double)xu0 * (double)xu0;
        lacc.mul(sg);
        clamped += wr.clamped ? 1 : 0;
        atomicAdd(vbar + iu, wu);
        xi_out[iu] = xu0;
        xibar_out[iu] = xbu;
        const unsigned long long slot = atomicAdd(rescue_count, 1ull);
        if (slot < rescue_cap) {
          rescue_rows[slot] = iu;
        } else {
          Row64<K> R;
          row_factor64<K, KT>(R, xs, row, k, xu, kf);
          const float s64 = (float)R.sigma;
          const double al = -(double)xbu / s64;
          const double sb = al * (double)xu0 + (double)nllbar / s64;
          row_backward64<K, KT>(R, xs, row, k, xu, kf, v, al, sb, s64, tl, ts, tn);
        }
      }
    }
    __syncwarp();
  }
  block_add3(tl * unit, ts, tn, thetabar);
  block_add_double(sq, acc);
  block_add_double(lacc.log_value(), acc + 1);
  unsigned long long c = clamped;
  for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(full, c, o);
  if (lane == 0 && c) atomicAdd(not_pd, c);
}

// The one-pass NLL value and gradient for 16 < k <= 32: eight lanes per point,
// as nll_grad_fused_kernel with the factor of pointoct.cuh.  Rows that need
// FP64 follow the others of their warp and are listed for
// factor_backward_rescue_kernel (the list holds every row).
template <int K, int KP, int KT>
__global__ void __launch_bounds__(kPairThreads, OctLayout<K>::kBlocks) nll_grad_fused_oct_kernel(
    const float4* __restrict__ xs, const int32_t* __restrict__ nbr, int64_t N, int k, int64_t n0,
    KernF kf, double unit, float nllbar, const float* __restrict__ v, float* vbar,
    float* __restrict__ xi_out, float* __restrict__ xibar_out, double* __restrict__ thetabar,
    double* __restrict__ acc, unsigned long long* __restrict__ not_pd, int64_t* __restrict__ rescue_rows,
    unsigned long long* __restrict__ rescue_count) {
  using OL = OctLayout<K>;
  extern __shared__ __align__(16) float psm[];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, r = lane & 7, first = (threadIdx.x >> 5) * 4;
  float* S = psm + (threadIdx.x >> 3) * OL::kStride;
  const uint64_t pol_v = l2_evict_last();
  LogAcc lacc;
  double sq = 0.0, tl = 0.0, ts = 0.0, tn = 0.0;
  unsigned long long clamped = 0;
  const int64_t npts = N - n0;
  const int64_t stride = (int64_t)gridDim.x * OL::kPoints;
  for (int64_t b0 = (int64_t)blockIdx.x * OL::kPoints; b0 < npts; b0 += stride) {
    __syncthreads();  // the warps of a block share the instruction stream
    const int64_t t = b0 + first + (lane >> 3);
    const bool valid = t < npts;
    const int64_t tt = valid ? t : npts - 1, i = n0 + tt;
    const int32_t* row = nbr + tt * KP;
    const float4 xq = __ldg(xs + i);
    oct_stage<K>(S, r, xs, row, KP);
    OctFactor<K> f;
    oct_factor<K, KT>(f, S, r, k, kf, xq);
    const bool rescue = valid && oct_needs_rescue(f, kf), act = valid && !rescue;
    float vv[K / 8];
    oct_gather<K, false>(vv, r, k, row, v, pol_v);
    const float sigma = f.sigma;
    const float xv = (ld_keep_f(v + i, pol_v) - oct_dot<K>(f.b, vv, S, r, KP)) / sigma;
    const float xb = nllbar * xv;
    const float w = xb / sigma;
    if (act) {
      if (r == 0) {
        sq += (double)xv * (double)xv;
        lacc.mul(sigma);
        clamped += f.clamped ? 1 : 0;
        atomicAdd(vbar + i, w);
      }
#pragma unroll
      for (int s = 0; s < K / 8; s++)
        if (8 * s + r < k && f.b[s] != 0.0f) atomicAdd(vbar + __ldg(row + 8 * s + r), f.b[s] * -w);
    }
    const float alpha = -xb / sigma;
    const float sigbar = alpha * xv + nllbar / sigma;
    oct_row_backward<K, KT>(f, S, r, k, kf, xq, vv, alpha, sigbar / (2.0f * sigma), act, tl, ts, tn);
    unsigned m = __ballot_sync(full, rescue) & 0x01010101u;
    while (m) {
      const int src = __ffs(m) - 1;
      m &= m - 1;
      __syncwarp();
      const int64_t u = b0 + first + (src >> 3), iu = n0 + u;
      const int32_t* ru = nbr + u * KP;
      const WarpRow64 wr = oct_row64<K, KT>(xs, ru, k, __ldg(xs + iu), kf,
                                         reinterpret_cast<double*>(psm + first * OL::kStride));
      const float b = lane < k ? (float)wr.b : 0.0f, sg = (float)wr.sigma;
      const float dot = warp_dot_stored_order<KP>(b, ru, v, pol_v);
      const float xu = __shfl_sync(full, (ld_keep_f(v + iu, pol_v) - dot) / sg, 0);
      const float xbu = nllbar * xu, wu = xbu / sg;
      if (lane < k && b != 0.0f) atomicAdd(vbar + ru[lane], b * -wu);
      if (lane == src) {
        sq += (double)xu * (double)xu;
        lacc.mul(sg);
        clamped += wr.clamped ? 1 : 0;
        atomicAdd(vbar + iu, wu);
        xi_out[iu] = xu;
        xibar_out[iu] = xbu;
        rescue_rows[atomicAdd(rescue_count, 1ull)] = iu;
      }
    }
    __syncwarp();
  }
  block_add3(tl * unit, ts, tn, thetabar);
  block_add_double(sq, acc);
  block_add_double(lacc.log_value(), acc + 1);
  unsigned long long c = clamped;
  for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(full, c, o);
  if (lane == 0 && c) atomicAdd(not_pd, c);
}

__global__ void scale_kernel(const float* __restrict__ x, float s, float* __restrict__ y,
                             int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    y[i] = s * x[i];
}

__global__ void mul_kernel(const float* __restrict__ a, const float* __restrict__ x,
                           float* __restrict__ y, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    y[i] = a[i] * x[i];
}

template <int K>
int launch_factor_backward_oct(graphgp_graph_t g, graphgp_factor_t f, int mode,
                               const float* coef, float beta, const float* v, const float* xi,
                               float* xibar, double* thetabar, const int32_t* nbr, int64_t N,
                               int64_t n0v, cudaStream_t s) {
  int64_t npts = N - n0v;
  if (npts <= 0) return GRAPHGP_OK;
  const unsigned grid = oct_grid<K>(npts);
  constexpr size_t smem = OctLayout<K>::kBytes;
  const KernF kf = make_kernf(f->kern, g);
  const double unit = graph_unit(g);
  Scratch sc(s);
  int64_t* rows = nullptr;
  unsigned long long* cnt = nullptr;
  GGP_TRY(sc.alloc(&rows, npts));
  GGP_TRY(sc.alloc(&cnt, 1));
  GGP_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), s));
  const unsigned rgrid = (unsigned)num_sms() * 2;
#define GGP_FB(KT)                                                                          \
  GGP_CUDA(allow_dyn_smem(factor_backward_oct_kernel<K, KT>, smem));                        \
  factor_backward_oct_kernel<K, KT><<<grid, kPairThreads, smem, s>>>(                       \
      g->xs, nbr, N, g->k, g->kp, n0v, kf, unit, mode, coef, beta, v, xi, xibar, thetabar, rows, cnt); \
  factor_backward_rescue_kernel<K, KT><<<rgrid, 128, 0, s>>>(                               \
      g->xs, nbr, g->k, g->kp, n0v, kf, unit, mode, coef, beta, v, xi, xibar, thetabar, rows, cnt, \
      (unsigned long long)npts)
  switch (f->kern.type) {
    case GRAPHGP_MATERN12: GGP_FB(GRAPHGP_MATERN12); break;
    case GRAPHGP_MATERN32: GGP_FB(GRAPHGP_MATERN32); break;
    case GRAPHGP_MATERN52: GGP_FB(GRAPHGP_MATERN52); break;
    default: GGP_FB(GRAPHGP_SQEXP); break;
  }
#undef GGP_FB
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

constexpr int64_t kBackwardRescueMax = 1 << 20;  // rows listed for the FP64 backward

template <int K>
int launch_factor_backward_pair(graphgp_graph_t g, graphgp_factor_t f, int mode,
                                  const float* coef, float beta, const float* v, const float* xi,
                                  float* xibar, double* thetabar, const int32_t* nbr,
                                  int64_t N, int64_t n0v, cudaStream_t s) {
  const int64_t npts = N - n0v;
  if (npts <= 0) return GRAPHGP_OK;
  const unsigned grid = pair_grid<K>(npts);
  const KernF kf = make_kernf(f->kern, g);
  const double unit = graph_unit(g);
  Scratch sc(s);
  const unsigned long long cap = (unsigned long long)std::min<int64_t>(npts, kBackwardRescueMax);
  int64_t* rows = nullptr;
  unsigned long long* cnt = nullptr;
  GGP_TRY(sc.alloc(&rows, cap));
  GGP_TRY(sc.alloc(&cnt, 1));
  GGP_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), s));
  const unsigned rgrid = (unsigned)num_sms() * 2;
  constexpr size_t smem = PairLayout<K>::kBytes;
#define GGP_FBT(KT)                                                                             \
  GGP_CUDA(allow_dyn_smem(factor_backward_pair_kernel<K, KT>, smem));                         \
  factor_backward_pair_kernel<K, KT><<<grid, kPairThreads, smem, s>>>(                        \
      g->xs, nbr, N, g->k, n0v, kf, unit, mode, coef, beta, v, xi, xibar, thetabar, rows, cnt, \
      cap);                                                                                     \
  factor_backward_rescue_kernel<K, KT><<<rgrid, 128, 0, s>>>(                                   \
      g->xs, nbr, g->k, g->kp, n0v, kf, unit, mode, coef, beta, v, xi, xibar, thetabar, rows, cnt, cap)
  switch (f->kern.type) {
    case GRAPHGP_MATERN12: GGP_FBT(GRAPHGP_MATERN12); break;
    case GRAPHGP_MATERN32: GGP_FBT(GRAPHGP_MATERN32); break;
    case GRAPHGP_MATERN52: GGP_FBT(GRAPHGP_MATERN52); break;
    default: GGP_FBT(GRAPHGP_SQEXP); break;
  }
#undef GGP_FBT
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

template <int K>
int launch_nll_grad_fused(graphgp_graph_t g, const graphgp_kernel* kern, float nllbar,
                          const float* v, float* vbar, float* xi_tmp, float* xibar_tmp,
                          double* thetabar, double* acc, unsigned long long* not_pd,
                          cudaStream_t s) {
  const int64_t npts = g->N - g->n0;
  if (npts <= 0) return GRAPHGP_OK;
  const unsigned grid = pair_grid<K>(npts);
  const KernF kf = make_kernf(*kern, g);
  const double unit = graph_unit(g);
  Scratch sc(s);
  const unsigned long long cap = (unsigned long long)std::min<int64_t>(npts, kBackwardRescueMax);
  int64_t* rows = nullptr;
  unsigned long long* cnt = nullptr;
  GGP_TRY(sc.alloc(&rows, cap));
  GGP_TRY(sc.alloc(&cnt, 1));
  GGP_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), s));
  const unsigned rgrid = (unsigned)num_sms() * 2;
  constexpr size_t smem = PairLayout<K>::kBytes;
#define GGP_NGF(KT)                                                                              \
  GGP_CUDA(allow_dyn_smem(nll_grad_fused_kernel<K, KT>, smem));                                  \
  nll_grad_fused_kernel<K, KT><<<grid, kPairThreads, smem, s>>>(                                 \
      g->xs, g->nbr, g->N, g->k, g->n0, kf, unit, nllbar, v, vbar, xi_tmp, xibar_tmp, thetabar, acc,  \
      not_pd, rows, cnt, cap);                                                                   \
  factor_backward_rescue_kernel<K, KT><<<rgrid, 128, 0, s>>>(                                    \
      g->xs, g->nbr, g->k, g->kp, g->n0, kf, unit, 0, xibar_tmp, nllbar, v, xi_tmp, nullptr, thetabar, \
      rows, cnt, cap)
  switch (kern->type) {
    case GRAPHGP_MATERN12: GGP_NGF(GRAPHGP_MATERN12); break;
    case GRAPHGP_MATERN32: GGP_NGF(GRAPHGP_MATERN32); break;
    case GRAPHGP_MATERN52: GGP_NGF(GRAPHGP_MATERN52); break;
    default: GGP_NGF(GRAPHGP_SQEXP); break;
  }
#undef GGP_NGF
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

template <int KP>
int launch_nll_grad_fused_oct(graphgp_graph_t g, const graphgp_kernel* kern, float nllbar,
                                const float* v, float* vbar, float* xi_tmp, float* xibar_tmp,
                                double* thetabar, double* acc, unsigned long long* not_pd,
                                cudaStream_t s) {
  const int64_t npts = g->N - g->n0;
  if (npts <= 0) return GRAPHGP_OK;
  constexpr int K = KP <= 24 ? 24 : 32;
  const unsigned grid = oct_grid<K>(npts);
  const KernF kf = make_kernf(*kern, g);
  const double unit = graph_unit(g);
  Scratch sc(s);
  int64_t* rows = nullptr;
  unsigned long long* cnt = nullptr;
  GGP_TRY(sc.alloc(&rows, npts));
  GGP_TRY(sc.alloc(&cnt, 1));
  GGP_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), s));
  const unsigned rgrid = (unsigned)num_sms() * 2;
  constexpr size_t smem = OctLayout<K>::kBytes;
#define GGP_NGG(KT)                                                                              \
  GGP_CUDA(allow_dyn_smem(nll_grad_fused_oct_kernel<K, KP, KT>, smem));                          \
  nll_grad_fused_oct_kernel<K, KP, KT><<<grid, kPairThreads, smem, s>>>(                         \
      g->xs, g->nbr, g->N, g->k, g->n0, kf, unit, nllbar, v, vbar, xi_tmp, xibar_tmp, thetabar, acc,  \
      not_pd, rows, cnt);                                                                        \
  factor_backward_rescue_kernel<K, KT><<<rgrid, 128, 0, s>>>(                                   \
      g->xs, g->nbr, g->k, g->kp, g->n0, kf, unit, 0, xibar_tmp, nllbar, v, xi_tmp, nullptr, thetabar, \
      rows, cnt, (unsigned long long)npts)
  switch (kern->type) {
    case GRAPHGP_MATERN12: GGP_NGG(GRAPHGP_MATERN12); break;
    case GRAPHGP_MATERN32: GGP_NGG(GRAPHGP_MATERN32); break;
    case GRAPHGP_MATERN52: GGP_NGG(GRAPHGP_MATERN52); break;
    default: GGP_NGG(GRAPHGP_SQEXP); break;
  }
#undef GGP_NGG
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

__global__ void nll_value_kernel(const double* __restrict__ acc, double* __restrict__ out) {
  out[0] = 0.5 * acc[0] + 0.5 * acc[1];
}

int launch_factor_backward_wide(graphgp_graph_t g, graphgp_factor_t f, int mode,
                                const float* coef, float beta, const float* v, const float* xi,
                                float* xibar, double* thetabar, const int32_t* nbr,
                                  int64_t N, int64_t n0v, cudaStream_t s) {
  const int64_t npts = N - n0v;
  if (npts <= 0) return GRAPHGP_OK;
  constexpr int kWarps = 4;
  const size_t smem = kWarps * sizeof(WideWarp);
  const unsigned grid = grid_for((npts + kWarps - 1) / kWarps * 128, 128, 4);
  const KernF kf = make_kernf(f->kern, g);
  const double unit = graph_unit(g);
  Scratch sc(s);
  int64_t* rows = nullptr;
  unsigned long long* cnt = nullptr;
  GGP_TRY(sc.alloc(&rows, npts));
  GGP_TRY(sc.alloc(&cnt, 1));
  GGP_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), s));
  const unsigned rgrid = (unsigned)num_sms() * 2;
#define GGP_FBW(KT)                                                                            \
  GGP_CUDA(cudaFuncSetAttribute(factor_backward_wide_kernel<KT>,                               \
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));      \
  factor_backward_wide_kernel<KT><<<grid, 32 * kWarps, smem, s>>>(                             \
      g->xs, nbr, N, g->k, g->kp, n0v, kf, unit, mode, coef, beta, v, xi, xibar, thetabar,   \
      rows, cnt);                                                                              \
  factor_backward_rescue_kernel<kWideK, KT><<<rgrid, 128, 0, s>>>(                             \
      g->xs, nbr, g->k, g->kp, n0v, kf, unit, mode, coef, beta, v, xi, xibar, thetabar, rows, cnt,  \
      (unsigned long long)npts)
  switch (f->kern.type) {
    case GRAPHGP_MATERN12: GGP_FBW(GRAPHGP_MATERN12); break;
    case GRAPHGP_MATERN32: GGP_FBW(GRAPHGP_MATERN32); break;
    case GRAPHGP_MATERN52: GGP_FBW(GRAPHGP_MATERN52); break;
    default: GGP_FBW(GRAPHGP_SQEXP); break;
  }
#undef GGP_FBW
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

int factor_backward_rows(graphgp_graph_t g, graphgp_factor_t f, int mode, const float* coef,
                         float beta, const float* v, const float* xi, float* xibar,
                         double* thetabar, int64_t t0, int64_t t1, cudaStream_t s) {
  if (t1 <= t0) return GRAPHGP_OK;
  const int32_t* nb = g->nbr + t0 * g->kp;
  const int64_t N = g->n0 + t1, n0v = g->n0 + t0;
  switch (g->kp) {
    case 4: return launch_factor_backward_pair<4>(g, f, mode, coef, beta, v, xi, xibar, thetabar, nb, N, n0v, s);
    case 8: return launch_factor_backward_pair<8>(g, f, mode, coef, beta, v, xi, xibar, thetabar, nb, N, n0v, s);
    case 12: return launch_factor_backward_pair<12>(g, f, mode, coef, beta, v, xi, xibar, thetabar, nb, N, n0v, s);
    case 16: return launch_factor_backward_pair<16>(g, f, mode, coef, beta, v, xi, xibar, thetabar, nb, N, n0v, s);
    case 20:
    case 24: return launch_factor_backward_oct<24>(g, f, mode, coef, beta, v, xi, xibar, thetabar, nb, N, n0v, s);
    case 28:
    case 32: return launch_factor_backward_oct<32>(g, f, mode, coef, beta, v, xi, xibar, thetabar, nb, N, n0v, s);
    default: return launch_factor_backward_wide(g, f, mode, coef, beta, v, xi, xibar, thetabar, nb, N, n0v, s);
  }
}

int factor_backward(graphgp_graph_t g, graphgp_factor_t f, int mode, const float* coef,
                    float beta, const float* v, const float* xi, float* xibar, double* thetabar,
                    cudaStream_t s) {
  return factor_backward_rows(g, f, mode, coef, beta, v, xi, xibar, thetabar, 0, g->N - g->n0, s);
}

}  // namespace

// Kbar_00 (n0 x n0, row-major, every entry a cotangent) of the dense block
// from u_0 and xi_0: Kbar = L0^-T Phi(L0^T Lbar0) L0^-1.
int dense_kbar(graphgp_graph_t g, graphgp_factor_t f, const float* u0, const float* xi0,
               float sgn, float ldbar, float* Kbar, cudaStream_t s) {
  int n0 = g->n0;
  int64_t nn = (int64_t)n0 * n0;
  Scratch sc(s);
  float *P = nullptr, *T = nullptr;
  GGP_TRY(sc.alloc(&P, nn));
  GGP_TRY(sc.alloc(&T, nn));
  unsigned grid = grid_for(nn, 256);
  dense_lbar_kernel<<<grid, 256, 0, s>>>(u0, xi0, f->L0, n0, sgn, ldbar, Kbar);
  const dim3 tiles((n0 + kGemmTile - 1) / kGemmTile, (n0 + kGemmTile - 1) / kGemmTile);
  dense_gemm_kernel<true, true><<<tiles, 256, 0, s>>>(f->L0, Kbar, P, n0);  // Phi(L0^T Lbar0)
  dense_gemm_kernel<true, false><<<tiles, 256, 0, s>>>(f->L0inv, P, T, n0);  // L0^-T P
  dense_gemm_kernel<false, false><<<tiles, 256, 0, s>>>(T, f->L0inv, Kbar, n0);  // (L0^-T P) L0^-1
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

namespace {

int dense_backward(graphgp_graph_t g, graphgp_factor_t f, const float* u0, const float* xi0,
                   float sgn, float ldbar, double* thetabar, cudaStream_t s) {
  int n0 = g->n0;
  int64_t nn = (int64_t)n0 * n0;
  Scratch sc(s);
  float* Lb = nullptr;
  GGP_TRY(sc.alloc(&Lb, nn));
  GGP_TRY(dense_kbar(g, f, u0, xi0, sgn, ldbar, Lb, s));
  unsigned grid = grid_for(nn, 256);
  const KernF kf = make_kernf(f->kern, g);
  const double unit = graph_unit(g);
  switch (f->kern.type) {
    case GRAPHGP_MATERN12: dense_theta_kernel<GRAPHGP_MATERN12><<<grid, 256, 0, s>>>(Lb, g->xs, n0, kf, unit, thetabar); break;
    case GRAPHGP_MATERN32: dense_theta_kernel<GRAPHGP_MATERN32><<<grid, 256, 0, s>>>(Lb, g->xs, n0, kf, unit, thetabar); break;
    case GRAPHGP_MATERN52: dense_theta_kernel<GRAPHGP_MATERN52><<<grid, 256, 0, s>>>(Lb, g->xs, n0, kf, unit, thetabar); break;
    default: dense_theta_kernel<GRAPHGP_SQEXP><<<grid, 256, 0, s>>>(Lb, g->xs, n0, kf, unit, thetabar); break;
  }
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

}  // namespace

int run_whiten_backward(graphgp_graph_t g, graphgp_factor_t f, const float* v, const float* xi,
                        const float* xibar, double logdetbar, float* vbar, double* thetabar,
                        cudaStream_t s) {
  int n0 = g->n0;
  // dense: vbar_0 = L0^-T xibar_0 (then children are subtracted below)
  dense_lower_tmatvec_kernel<false><<<(n0 + 31) / 32, 256, 0, s>>>(f->L0inv, xibar, vbar, n0);
  GGP_CUDA(cudaGetLastError());
  if (thetabar) GGP_TRY(dense_backward(g, f, vbar, xi, -1.0f, (float)logdetbar, thetabar, s));
  if (g->N > n0) {
    GGP_CUDA(cudaMemsetAsync(vbar + n0, 0, (g->N - n0) * sizeof(float), s));
    GGP_TRY(whiten_adjoint_scatter(g, f, xibar, vbar, n0, g->N, s));
  }
  if (thetabar)
    GGP_TRY(factor_backward(g, f, 0, xibar, (float)(2.0 * logdetbar), v, xi, nullptr, thetabar, s));
  return GRAPHGP_OK;
}

int run_generate_backward(graphgp_graph_t g, graphgp_factor_t f, const float* xi, const float* v,
                          const float* vbar, float* xibar, double* thetabar, cudaStream_t s) {
  float* u = g->tmp_vec;
  int n0 = g->n0;
  GGP_CUDA(cudaMemcpyAsync(u, vbar, g->N * sizeof(float), cudaMemcpyDeviceToDevice, s));
  const std::vector<int64_t>& lo = g->level_off_h;
  const int32_t* nb = g->nbr;
  const float* bw = f->b;
  const int64_t* lod = g->level_off_d;
  int nl = g->num_levels, head = 1;  // levels [1, head) to one block
  int64_t n0l = n0;
  while (head < nl && head < kHeadLevels && (lo[head + 1] - lo[head]) * g->kp <= kHeadEntries &&
         lo[head + 1] <= kHeadPoints)
    head++;
  if (head < nl) {
    GGP_CUDA(cudaMemsetAsync(g->level_bar, 0, g->num_levels * sizeof(uint32_t), s));
    LevelBarrier lb{g->level_bar, g->err, g->max_spin};
    void* args[] = {(void*)&nb, (void*)&bw, (void*)&u, (void*)&lod, (void*)&head, (void*)&nl,
                    (void*)&n0l, (void*)&lb};
#define GGP_GSC(KP)                                                                              \
  {                                                                                              \
    static int max_grid_dev[kMaxDevices] = {};                                                   \
    const int max_grid = coop_grid_cached(max_grid_dev, generate_adjoint_scatter_kernel<KP>, 256); \
    const int grid = (int)std::min<int64_t>(max_grid, std::max<int64_t>((g->max_level_size + 63) / 64, 1)); \
    GGP_CUDA(cudaLaunchCooperativeKernel((const void*)generate_adjoint_scatter_kernel<KP>,       \
                                         dim3(grid), dim3(256), args, 0, s));                    \
  }
    GGP_ADJ_KP_DISPATCH(g->kp, GGP_GSC);
#undef GGP_GSC
  }
  if (head > 1) {
    const size_t smem = (size_t)lo[head] * sizeof(float) + (head + 1) * sizeof(int32_t);
#define GGP_GSH(KP)                                                                         \
  {                                                                                         \
    GGP_CUDA(allow_dyn_smem(generate_adjoint_head_kernel<KP>, smem));                       \
    generate_adjoint_head_kernel<KP><<<1, kHeadThreads, smem, s>>>(nb, bw, u, lod, head, n0l); \
  }
    GGP_ADJ_KP_DISPATCH(g->kp, GGP_GSH);
#undef GGP_GSH
    GGP_CUDA(cudaGetLastError());
  }
  // dense: xibar_0 = L0^T u_0, Lbar0 = tril(u_0 xi_0^T)
  dense_lower_tmatvec_kernel<false><<<(n0 + 31) / 32, 256, 0, s>>>(f->L0, u, xibar, n0);
  GGP_CUDA(cudaGetLastError());
  if (!thetabar) {  // vector cotangent only: xibar_i = sigma_i u_i
    if (g->N > n0)
      mul_kernel<<<grid_for(g->N - n0, 256), 256, 0, s>>>(f->sigma + n0, u + n0, xibar + n0,
                                                           g->N - n0);
    GGP_CUDA(cudaGetLastError());
    return GRAPHGP_OK;
  }
  GGP_TRY(dense_backward(g, f, u, xi, 1.0f, 0.0f, thetabar, s));
  GGP_TRY(factor_backward(g, f, 1, u, 0.0f, v, xi, xibar, thetabar, s));
  return GRAPHGP_OK;
}

int run_whiten(graphgp_graph_t g, graphgp_factor_t f, const float* v, float* xi, double* sq,
               cudaStream_t s);

// ---- row ranges (sharding by position range) ---------------------------------
// The NLL and its gradient restricted to the positions [p0, p1) whose factor a
// row-range handle holds: the sums over disjoint ranges add up to the whole.

// sum_e b_e v[c_e] of one row in the stored sweeps' order (gen_lanes slices,
// two alternating accumulators per slice, slices combined as their xor
// shuffles do), so xi is bit-identical to the whiten sweep's.
__device__ __forceinline__ float row_dot_stored_order(const float* __restrict__ b,
                                                      const int32_t* __restrict__ c, int kp,
                                                      const float* __restrict__ v) {
  const int lanes = gen_lanes(kp), hp = kp / lanes;
  float part[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  for (int h = 0; h < lanes; h++) {
    float acc0 = 0.0f, acc1 = 0.0f;
    for (int e = h * hp; e < (h + 1) * hp; e += 4) {
      acc0 = fmaf(b[e], v[c[e]], acc0);
      acc1 = fmaf(b[e + 1], v[c[e + 1]], acc1);
      acc0 = fmaf(b[e + 2], v[c[e + 2]], acc0);
      acc1 = fmaf(b[e + 3], v[c[e + 3]], acc1);
    }
    part[h] = acc0 + acc1;
  }
  if (lanes == 4) return (part[0] + part[2]) + (part[1] + part[3]);
  if (lanes == 2) return part[0] + part[1];
  return part[0];
}

// xi_i = (v_i - b_i . v_c(i)) / sigma_i for rows t in [t0, t1); optional FP64
// sum of xi_i^2 (added to *sq).
__global__ void whiten_rows_kernel(const int32_t* __restrict__ nbr, const float* __restrict__ b,
                                   const float* __restrict__ sigma, const float* __restrict__ v,
                                   float* __restrict__ xi, int kp, int64_t n0, int64_t t0,
                                   int64_t t1, double* __restrict__ sq) {
  double local = 0.0;
  for (int64_t t = t0 + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < t1;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = n0 + t;
    const float acc = row_dot_stored_order(b + t * kp, nbr + t * kp, kp, v);
    const float out = (v[i] - acc) / sigma[i];
    xi[i] = out;
    local += (double)out * (double)out;
  }
  if (sq) block_add_double(local, sq);
}

__global__ void nll_rows_finish_kernel(const double* __restrict__ sq,
                                       const double* __restrict__ logdet,
                                       double* __restrict__ out) {
  out[0] = 0.5 * sq[0] + 0.5 * logdet[0];
}

// xi over the factor's positions into xi (full length; other entries untouched).
int whiten_rows(graphgp_graph_t g, graphgp_factor_t f, const float* v, float* xi, double* sq,
                cudaStream_t s) {
  const int64_t p0 = f->row_begin, p1 = f->row_end;
  if (p0 == 0) GGP_TRY(dense_matvec(f->L0inv, v, xi, g->n0, sq, s));
  const int64_t t0 = std::max<int64_t>(p0, g->n0) - g->n0, t1 = p1 - g->n0;
  if (t1 > t0) {
    whiten_rows_kernel<<<grid_for(t1 - t0, 256), 256, 0, s>>>(g->nbr, f->b, f->sigma, v, xi, g->kp,
                                                              g->n0, t0, t1, sq);
    GGP_CUDA(cudaGetLastError());
  }
  return GRAPHGP_OK;
}

}  // namespace ggp

using namespace ggp;

static bool rows_ok(graphgp_graph_t g, graphgp_factor_t f) {
  return g && f && f->g == g && f->row_end >= 0;
}

extern "C" int graphgp_nll_rows(graphgp_graph_t g, graphgp_factor_t f, const float* v_d,
                                double* out_d, void* stream) {
  if (!rows_ok(g, f) || !v_d || !out_d) return GRAPHGP_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  Scratch sc(s);
  double* sq = nullptr;
  GGP_TRY(sc.alloc(&sq, 1));
  GGP_CUDA(cudaMemsetAsync(sq, 0, sizeof(double), s));
  GGP_TRY(whiten_rows(g, f, v_d, g->tmp_vec2, sq, s));
  nll_rows_finish_kernel<<<1, 1, 0, s>>>(sq, f->logdet, out_d);
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

extern "C" int graphgp_nll_backward_rows(graphgp_graph_t g, graphgp_factor_t f, const float* v_d,
                                         double nllbar, float* vbar_d, double* thetabar_d,
                                         void* stream) {
  if (!rows_ok(g, f) || !v_d || !vbar_d || !thetabar_d) return GRAPHGP_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  float* xi = g->tmp_vec2;
  float* xibar = g->tmp_vec;
  GGP_TRY(whiten_rows(g, f, v_d, xi, nullptr, s));
  scale_kernel<<<grid_for(g->N, 256), 256, 0, s>>>(xi, (float)nllbar, xibar, g->N);
  GGP_CUDA(cudaGetLastError());
  const int n0 = g->n0;
  const int64_t p0 = f->row_begin, p1 = f->row_end;
  if (p0 == 0) {
    // dense rows: u_0 = L0^-T xibar_0 into vbar_0, and the dense block's theta part
    Scratch sc(s);
    float* u0 = nullptr;
    GGP_TRY(sc.alloc(&u0, n0));
    dense_lower_tmatvec_kernel<false><<<(n0 + 31) / 32, 256, 0, s>>>(f->L0inv, xibar, u0, n0);
    dense_lower_tmatvec_kernel<true><<<(n0 + 31) / 32, 256, 0, s>>>(f->L0inv, xibar, vbar_d, n0);
    GGP_CUDA(cudaGetLastError());
    GGP_TRY(dense_backward(g, f, u0, xi, -1.0f, (float)(0.5 * nllbar), thetabar_d, s));
  }
  const int64_t t0 = std::max<int64_t>(p0, n0) - n0, t1 = p1 - n0;
  if (t1 > t0) {
    // the neighbours of a range belong to other rows and ranges: atomic adds
    GGP_TRY(whiten_adjoint_scatter(g, f, xibar, vbar_d, n0 + t0, n0 + t1, s));
    GGP_TRY(factor_backward_rows(g, f, 0, xibar, (float)nllbar, v_d, xi, nullptr, thetabar_d, t0,
                                 t1, s));
  }
  return GRAPHGP_OK;
}


static bool pair_ok(graphgp_graph_t g, graphgp_factor_t f) {
  return g && f && f->g == g && f->row_end < 0;
}

extern "C" int graphgp_generate_backward(graphgp_graph_t g, graphgp_factor_t f, const float* xi_d,
                                         const float* v_d, const float* vbar_d, float* xibar_d,
                                         double* thetabar_d, void* stream) {
  if (!pair_ok(g, f) || !xi_d || !v_d || !vbar_d || !xibar_d) return GRAPHGP_ERR_INVALID;
  return run_generate_backward(g, f, xi_d, v_d, vbar_d, xibar_d, thetabar_d, (cudaStream_t)stream);
}

extern "C" int graphgp_whiten_backward(graphgp_graph_t g, graphgp_factor_t f, const float* v_d,
                                       const float* xi_d, const float* xibar_d, double logdetbar,
                                       float* vbar_d, double* thetabar_d, void* stream) {
  if (!pair_ok(g, f) || !xi_d || !v_d || !xibar_d || !vbar_d) return GRAPHGP_ERR_INVALID;
  return run_whiten_backward(g, f, v_d, xi_d, xibar_d, logdetbar, vbar_d, thetabar_d,
                             (cudaStream_t)stream);
}

extern "C" int graphgp_nll_backward(graphgp_graph_t g, graphgp_factor_t f, const float* v_d,
                                    double nllbar, float* vbar_d, double* thetabar_d,
                                    void* stream) {
  if (!pair_ok(g, f) || !v_d || !vbar_d) return GRAPHGP_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  float* xi = g->tmp_vec2;
  float* xibar = g->tmp_vec;
  GGP_TRY(run_whiten(g, f, v_d, xi, nullptr, s));
  scale_kernel<<<grid_for(g->N, 256), 256, 0, s>>>(xi, (float)nllbar, xibar, g->N);
  GGP_CUDA(cudaGetLastError());
  return run_whiten_backward(g, f, v_d, xi, xibar, 0.5 * nllbar, vbar_d, thetabar_d, s);
}

// NLL value and gradient with the factors recomputed in the pass (the
// on-the-fly form of graphgp_nll + graphgp_nll_backward).
extern "C" int graphgp_nll_grad_fused(graphgp_graph_t g, const graphgp_kernel* kern,
                                      const float* v_d, double nllbar, double* nll_d,
                                      float* vbar_d, double* thetabar_d, uint64_t* not_pd_d,
                                      void* stream) {
  if (!g || !valid_kernel(kern) || g->k > 32 || !v_d || !nll_d || !vbar_d || !thetabar_d)
    return GRAPHGP_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  unsigned long long* bad = (unsigned long long*)not_pd_d;
  Scratch sc(s);
  double* acc = nullptr;  // [0] xi.xi, [1] logdet
  GGP_TRY(sc.alloc(&acc, 2));
  GGP_CUDA(cudaMemsetAsync(acc, 0, 16, s));
  if (!bad) {
    GGP_TRY(sc.alloc(&bad, 1));
    GGP_CUDA(cudaMemsetAsync(bad, 0, 8, s));
  }
  const int n0 = g->n0;
  float* xi = g->tmp_vec2;  // xi_0 and the FP64 rows' xi
  float* xb = g->tmp_vec;   // nllbar xi for the same positions
  graphgp_factor_s f;
  GGP_TRY(dense_into(g, kern, sc, acc + 1, bad, f, s));
  GGP_TRY(dense_matvec(f.L0inv, v_d, xi, n0, acc, s));
  scale_kernel<<<(n0 + 255) / 256, 256, 0, s>>>(xi, (float)nllbar, xb, n0);
  dense_lower_tmatvec_kernel<false><<<(n0 + 31) / 32, 256, 0, s>>>(f.L0inv, xb, vbar_d, n0);
  GGP_CUDA(cudaGetLastError());
  GGP_TRY(dense_backward(g, &f, vbar_d, xi, -1.0f, (float)(0.5 * nllbar), thetabar_d, s));
  if (g->N > n0) {
    GGP_CUDA(cudaMemsetAsync(vbar_d + n0, 0, (g->N - n0) * sizeof(float), s));
    int rc = GRAPHGP_OK;
    switch (g->kp) {
      case 4: rc = launch_nll_grad_fused<4>(g, kern, (float)nllbar, v_d, vbar_d, xi, xb, thetabar_d, acc, bad, s); break;
      case 8: rc = launch_nll_grad_fused<8>(g, kern, (float)nllbar, v_d, vbar_d, xi, xb, thetabar_d, acc, bad, s); break;
      case 12: rc = launch_nll_grad_fused<12>(g, kern, (float)nllbar, v_d, vbar_d, xi, xb, thetabar_d, acc, bad, s); break;
      case 16: rc = launch_nll_grad_fused<16>(g, kern, (float)nllbar, v_d, vbar_d, xi, xb, thetabar_d, acc, bad, s); break;
      case 20: rc = launch_nll_grad_fused_oct<20>(g, kern, (float)nllbar, v_d, vbar_d, xi, xb, thetabar_d, acc, bad, s); break;
      case 24: rc = launch_nll_grad_fused_oct<24>(g, kern, (float)nllbar, v_d, vbar_d, xi, xb, thetabar_d, acc, bad, s); break;
      case 28: rc = launch_nll_grad_fused_oct<28>(g, kern, (float)nllbar, v_d, vbar_d, xi, xb, thetabar_d, acc, bad, s); break;
      default: rc = launch_nll_grad_fused_oct<32>(g, kern, (float)nllbar, v_d, vbar_d, xi, xb, thetabar_d, acc, bad, s); break;
    }
    GGP_TRY(rc);
  }
  nll_value_kernel<<<1, 1, 0, s>>>(acc, nll_d);
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}
