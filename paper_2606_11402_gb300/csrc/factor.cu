// Per-point conditioning factors (Sec. 2.1 Eq. 2; Alg. 1).  The dense initial
// block is in dense.cu.
//
// Per point i with c = c(i): b_i = K_ic K_cc^-1 and sigma_i^2 =
// K_ii - K_ic K_cc^-1 K_ci, two lanes per point for k <= 16 (pointpair.cuh),
// eight for k <= 32 (pointoct.cuh), a warp above (pointwide.cuh).  Pivots below
// 1e-7 of their diagonal entry are raised to that floor and counted.  logdet =
// sum log sigma_i^2 is reduced in FP64 from the stored FP32 sigma (a running
// FP64 product with separate exponent, one log per thread).
#include "pointoct.cuh"
#include "pointwide.cuh"

namespace ggp {
namespace {

// Rows whose FP32 factor needs the FP64 rescue (rescue.cuh) are listed here
// and recomputed afterwards (k <= 32: factor_rescue_group_kernel, several rows
// per warp; above: factor_rescue_kernel, one thread per row), so that a warp
// does not stall on the FP64 row of one of its points.  A row
// that finds the list full is recomputed in place.
struct RescueList {
  int64_t* rows;
  unsigned long long* count;
  unsigned long long cap;
  __device__ __forceinline__ bool defer(int64_t i) const {
    const unsigned long long slot = atomicAdd(count, 1ull);
    if (slot < cap) {
      rows[slot] = i;
      return true;
    }
    return false;
  }
};

// The rows [t0, t1) of the sparse positions, seen by the factor kernels as a
// graph of their own: positions n0 + t0 .. n0 + t1 - 1, neighbour and weight
// rows shifted by t0 (position indices stay global).
struct RowView {
  const int32_t* nbr;
  float* b;
  int64_t N, n0;
};

// 16 < k <= 32: eight lanes per point (pointoct.cuh), K = 24 or 32.
template <int K, int KT>
__global__ void __launch_bounds__(kPairThreads, OctLayout<K>::kBlocks) point_factor_oct_kernel(
    const float4* __restrict__ xs, const int32_t* __restrict__ nbr, int64_t N, int k, int kp,
    int64_t n0, KernF kf, float* __restrict__ b_out, float* __restrict__ sigma_out,
    double* __restrict__ logdet, unsigned long long* __restrict__ not_pd, RescueList rl) {
  using OL = OctLayout<K>;
  extern __shared__ __align__(16) float psm[];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, r = lane & 7, first = (threadIdx.x >> 5) * 4;
  float* S = psm + (threadIdx.x >> 3) * OL::kStride;
  LogAcc acc;
  unsigned long long clamped_rows = 0;
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
    bool deferred = false;
    if (rescue && r == 0) deferred = rl.defer(i);
    deferred = __shfl_sync(full, deferred, 0, 8);
    oct_rescue<K, KT>(f, rescue && !deferred, psm + first * OL::kStride, r, xs, row, k, xq, kf);
    if (valid && !deferred) {  // (a row that found the list full is recomputed by now)
#pragma unroll
      for (int s = 0; s < K / 8; s++)
        if (8 * s + r < kp) b_out[tt * kp + 8 * s + r] = 8 * s + r < k ? f.b[s] : 0.0f;
      if (r == 0) {
        sigma_out[i] = f.sigma;
        acc.mul(f.sigma);
        if (f.clamped) clamped_rows++;
      }
    }
  }
  block_add_double(acc.log_value(), logdet);
  for (int o = 16; o; o >>= 1) clamped_rows += __shfl_xor_sync(full, clamped_rows, o);
  if (lane == 0 && clamped_rows) atomicAdd(not_pd, clamped_rows);
}

// k <= 16 (K = padded row length): two lanes per point (pointpair.cuh).
template <int K, int KT>
__global__ void __launch_bounds__(kPairThreads, PairLayout<K>::kBlocks) point_factor_pair_kernel(
    const float4* __restrict__ xs, const int32_t* __restrict__ nbr, int64_t N, int k, int64_t n0,
    KernF kf, float* __restrict__ b_out, float* __restrict__ sigma_out,
    double* __restrict__ logdet, unsigned long long* __restrict__ not_pd, RescueList rl) {
  using PL = PairLayout<K>;
  extern __shared__ __align__(16) float psm[];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, r = lane & 1;
  float* S = psm + (threadIdx.x >> 1) * PL::kStride;
  LogAcc acc;
  unsigned long long clamped_rows = 0;
  const int64_t npts = N - n0;
  const int64_t stride = (int64_t)gridDim.x * PL::kPoints;
  const int first = (threadIdx.x >> 5) * 16;
  // the next point's indices and coordinates are loaded while this one's
  // factor ends
  PairLoad<K> ld;
  float4 xn;
  int64_t b0 = (int64_t)blockIdx.x * PL::kPoints;
  auto at = [&](int64_t blk) { return min(blk + first + (lane >> 1), npts - 1); };
  ld.indices(r, nbr + at(b0) * K);
  ld.coords(r, xs);
  xn = __ldg(xs + n0 + at(b0));
  for (; b0 < npts; b0 += stride) {
    // The block's warps start each point together: the straight-line code is
    // longer than the instruction caches, and warps in step share its fetches
    // (2^23 rows at K = 16: 3.65 -> 3.45 ms).
    __syncthreads();
    const int64_t base = b0 + first, t = base + (lane >> 1);
    const bool valid = t < npts;
    const int64_t i = n0 + (valid ? t : 0);
    const float4 xq = xn;
    ld.stage(S, r);
    PairFactor<K> f;
    pair_factor<K, KT>(
        f, S, r, k, kf, xq, [&] { ld.indices(r, nbr + at(b0 + stride) * K); },
        [&] {
          ld.coords(r, xs);
          xn = __ldg(xs + n0 + at(b0 + stride));
        });
    bool rescue = valid && pair_needs_rescue(f, kf), deferred = false;
    if (rescue && r == 0) deferred = rl.defer(i);
    deferred = __shfl_sync(full, deferred, 0, 2);
    if (valid && !rescue) {
      float4* bo = reinterpret_cast<float4*>(b_out + t * K);
#pragma unroll
      for (int q = 0; q < (K + 4) / 8; q++) {
        const int c0 = 2 * q, c1 = 2 * q + 1 < K / 4 ? 2 * q + 1 : 2 * q;
        const float2 u = r ? f.b[2 * c1] : f.b[2 * c0], w = r ? f.b[2 * c1 + 1] : f.b[2 * c0 + 1];
        if (2 * q + r < K / 4) bo[2 * q + r] = make_float4(u.x, u.y, w.x, w.y);
      }
      if (r == 0) {
        sigma_out[i] = f.sigma;
        acc.mul(f.sigma);
        if (f.clamped) clamped_rows++;
      }
    }
    // the list is full: the warp recomputes such rows here, one at a time
    unsigned m = __ballot_sync(full, rescue && !deferred && r == 0);
    while (m) {
      const int src = __ffs(m) - 1;
      m &= m - 1;
      __syncwarp();
      const int64_t u = base + (src >> 1);
      double* W = reinterpret_cast<double*>(psm + first * PL::kStride);
      const WarpRow64 w = warp_row_factor64<K, KT>(xs, nbr + u * K, k, __ldg(xs + n0 + u), kf, W);
      if (lane < K) b_out[u * K + lane] = lane < k ? (float)w.b : 0.0f;
      if (lane == src) {
        const float sg = (float)w.sigma;
        sigma_out[i] = sg;
        acc.mul(sg);
        if (w.clamped) clamped_rows++;
      }
    }
  }
  block_add_double(acc.log_value(), logdet);
  for (int o = 16; o; o >>= 1) clamped_rows += __shfl_xor_sync(full, clamped_rows, o);
  if (lane == 0 && clamped_rows) atomicAdd(not_pd, clamped_rows);
}

// 32 < k <= 64: one warp per point with the factor in shared memory
// (pointwide.cuh).  Rows that need the FP64 rescue are recomputed by lane 0.
template <int KT>
__global__ void __launch_bounds__(128) point_factor_wide_kernel(
    const float4* __restrict__ xs, const int32_t* __restrict__ nbr, int64_t N, int k, int kp,
    int64_t n0, KernF kf, float* __restrict__ b_out, float* __restrict__ sigma_out,
    double* __restrict__ logdet, unsigned long long* __restrict__ not_pd, RescueList rl) {
  extern __shared__ __align__(16) unsigned char wide_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  WideWarp& W = reinterpret_cast<WideWarp*>(wide_smem)[warp];
  LogAcc acc;
  unsigned long long clamped_rows = 0;
  const int64_t npts = N - n0;
  const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + warp; t < npts; t += nw) {
    const int64_t i = n0 + t;
    const int32_t* row = nbr + t * kp;
    for (int a = lane; a < k; a += 32) W.x[a] = __ldg(xs + row[a]);
    __syncwarp();
    const float4 xq = __ldg(xs + i);
    WideFactor r = point_factor_wide<KT>(W, k, kf, xq);
    if (wide_needs_rescue(W, r, k, kf)) {
      bool deferred = false;
      if (lane == 0) deferred = rl.defer(i);
      if (__shfl_sync(0xffffffffu, deferred, 0)) continue;
      if (lane == 0) {
        Row64<kWideK> R;
        row_factor64<kWideK, KT>(R, xs, row, k, xq, kf);
        for (int e = 0; e < kp; e++) b_out[t * kp + e] = e < k ? (float)R.b[e] : 0.0f;
        const float sg = (float)R.sigma;
        sigma_out[i] = sg;
        acc.mul(sg);
        if (R.clamped) clamped_rows++;
      }
    } else {
      for (int a = lane; a < kp; a += 32) b_out[t * kp + a] = a < k ? W.y[a] : 0.0f;
      if (lane == 0) {
        sigma_out[i] = r.sigma;
        acc.mul(r.sigma);
        if (r.clamped) clamped_rows++;
      }
    }
    __syncwarp();
  }
  double lv = (lane == 0) ? acc.log_value() : 0.0;
  block_add_double(lv, logdet);
  for (int o = 16; o; o >>= 1) clamped_rows += __shfl_xor_sync(0xffffffffu, clamped_rows, o);
  if (lane == 0 && clamped_rows) atomicAdd(not_pd, clamped_rows);
}

// The FP64 rows listed by the factor kernels: b (row stride kp), sigma, and
// their log-determinant and floor counts.
// k <= 32: several rows per warp (group_row_factor64).
constexpr int kRescueWarps = 4;

template <int KMAX, int KT>
__global__ void __launch_bounds__(32 * kRescueWarps) factor_rescue_group_kernel(
    const float4* __restrict__ xs, const int32_t* __restrict__ nbr, int k, int kp, int64_t n0,
    KernF kf, RescueList rl, float* __restrict__ b_out, float* __restrict__ sigma_out,
    double* __restrict__ logdet, unsigned long long* __restrict__ not_pd) {
  using GR = GroupRow64<KMAX>;
  extern __shared__ __align__(16) unsigned char rsm[];
  const int lane = threadIdx.x & 31, grp = threadIdx.x / GR::G, g = threadIdx.x % GR::G;
  GR& R = reinterpret_cast<GR*>(rsm)[grp];
  LogAcc acc;
  unsigned long long clamped_rows = 0;
  const unsigned long long cnt = *rl.count;
  const int64_t n = (int64_t)(cnt < rl.cap ? cnt : rl.cap);
  constexpr int kPerBlock = kRescueWarps * GR::kRows;
  const int64_t wrow = (threadIdx.x >> 5) * GR::kRows;  // the warp's first row in the block's
  for (int64_t r0 = (int64_t)blockIdx.x * kPerBlock + wrow; r0 < n;
       r0 += (int64_t)gridDim.x * kPerBlock) {  // the same on every lane
    const int64_t r = r0 + lane / GR::G;
    const bool act = r < n;
    const int64_t i = act ? rl.rows[r] : n0, t = i - n0;
    bool clamped;
    const double sigma = group_row_factor64<KMAX, KT>(R, act, xs, nbr + t * kp, k, __ldg(xs + i), kf,
                                                      clamped);
    if (act) {
      for (int a = g; a < kp; a += GR::G) b_out[t * kp + a] = a < k ? (float)R.y[a] : 0.0f;
      if (g == 0) {
        const float sg = (float)sigma;
        sigma_out[i] = sg;
        acc.mul(sg);
        if (clamped) clamped_rows++;
      }
    }
  }
  block_add_double(acc.log_value(), logdet);
  for (int o = 16; o; o >>= 1) clamped_rows += __shfl_xor_sync(0xffffffffu, clamped_rows, o);
  if (lane == 0 && clamped_rows) atomicAdd(not_pd, clamped_rows);
}

// k > 32: one thread per listed row.
template <int KMAX, int KT>
__global__ void __launch_bounds__(128) factor_rescue_kernel(
    const float4* __restrict__ xs, const int32_t* __restrict__ nbr, int k, int kp, int64_t n0,
    KernF kf, RescueList rl, float* __restrict__ b_out, float* __restrict__ sigma_out,
    double* __restrict__ logdet, unsigned long long* __restrict__ not_pd) {
  LogAcc acc;
  unsigned long long clamped_rows = 0;
  const unsigned long long cnt = *rl.count;
  const int64_t n = (int64_t)(cnt < rl.cap ? cnt : rl.cap);
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = rl.rows[r];
    const int64_t t = i - n0;
    Row64<KMAX> R;
    row_factor64<KMAX, KT>(R, xs, nbr + t * kp, k, __ldg(xs + i), kf);
    for (int e = 0; e < kp; e++) b_out[t * kp + e] = e < k ? (float)R.b[e] : 0.0f;
    const float sg = (float)R.sigma;
    sigma_out[i] = sg;
    acc.mul(sg);
    if (R.clamped) clamped_rows++;
  }
  block_add_double(acc.log_value(), logdet);
  for (int o = 16; o; o >>= 1) clamped_rows += __shfl_xor_sync(0xffffffffu, clamped_rows, o);
  if ((threadIdx.x & 31) == 0 && clamped_rows) atomicAdd(not_pd, clamped_rows);
}

template <int KMAX>
int launch_rescue(int type, graphgp_graph_t g, graphgp_factor_t f, const KernF& kf,
                  const RescueList& rl, const RowView& rv, cudaStream_t s) {
  const unsigned grid = 4 * (unsigned)num_sms();
#define GGP_RS(KT)                                                                          \
  if constexpr (KMAX <= 32) {                                                               \
    constexpr size_t smem = kRescueWarps * GroupRow64<KMAX>::kRows * sizeof(GroupRow64<KMAX>); \
    GGP_CUDA(allow_dyn_smem(factor_rescue_group_kernel<KMAX, KT>, smem));                   \
    factor_rescue_group_kernel<KMAX, KT><<<grid, 32 * kRescueWarps, smem, s>>>(             \
        g->xs, rv.nbr, g->k, g->kp, rv.n0, kf, rl, rv.b, f->sigma, f->logdet, f->not_pd);   \
  } else {                                                                                  \
    factor_rescue_kernel<KMAX, KT><<<grid, 128, 0, s>>>(                                    \
        g->xs, rv.nbr, g->k, g->kp, rv.n0, kf, rl, rv.b, f->sigma, f->logdet, f->not_pd);   \
  }
  switch (type) {
    case GRAPHGP_MATERN12: GGP_RS(GRAPHGP_MATERN12); break;
    case GRAPHGP_MATERN32: GGP_RS(GRAPHGP_MATERN32); break;
    case GRAPHGP_MATERN52: GGP_RS(GRAPHGP_MATERN52); break;
    default: GGP_RS(GRAPHGP_SQEXP); break;
  }
#undef GGP_RS
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

template <int K>
int launch_point_oct(int type, graphgp_graph_t g, graphgp_factor_t f, const KernF& kf,
                     const RescueList& rl, const RowView& rv, cudaStream_t s) {
  const unsigned grid = oct_grid<K>(rv.N - rv.n0);
  constexpr size_t smem = OctLayout<K>::kBytes;
#define GGP_PF(KT)                                                                             \
  GGP_CUDA(allow_dyn_smem(point_factor_oct_kernel<K, KT>, smem));                              \
  point_factor_oct_kernel<K, KT><<<grid, kPairThreads, smem, s>>>(                             \
      g->xs, rv.nbr, rv.N, g->k, g->kp, rv.n0, kf, rv.b, f->sigma, f->logdet, f->not_pd, rl)
  switch (type) {
    case GRAPHGP_MATERN12: GGP_PF(GRAPHGP_MATERN12); break;
    case GRAPHGP_MATERN32: GGP_PF(GRAPHGP_MATERN32); break;
    case GRAPHGP_MATERN52: GGP_PF(GRAPHGP_MATERN52); break;
    default: GGP_PF(GRAPHGP_SQEXP); break;
  }
#undef GGP_PF
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

template <int K>
int launch_point_pair(int type, graphgp_graph_t g, graphgp_factor_t f, const KernF& kf,
                      const RescueList& rl, const RowView& rv, cudaStream_t s) {
  const int64_t npts = rv.N - rv.n0;
  const unsigned grid = pair_grid<K>(npts);
  constexpr size_t smem = PairLayout<K>::kBytes;
#define GGP_PT(KT)                                                                            \
  GGP_CUDA(allow_dyn_smem(point_factor_pair_kernel<K, KT>, smem));                            \
  point_factor_pair_kernel<K, KT><<<grid, kPairThreads, smem, s>>>(                           \
      g->xs, rv.nbr, rv.N, g->k, rv.n0, kf, rv.b, f->sigma, f->logdet, f->not_pd, rl)
  switch (type) {
    case GRAPHGP_MATERN12: GGP_PT(GRAPHGP_MATERN12); break;
    case GRAPHGP_MATERN32: GGP_PT(GRAPHGP_MATERN32); break;
    case GRAPHGP_MATERN52: GGP_PT(GRAPHGP_MATERN52); break;
    default: GGP_PT(GRAPHGP_SQEXP); break;
  }
#undef GGP_PT
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

constexpr int kWideWarps = 4;  // warps per block of the wide kernels
constexpr int64_t kRescueListMax = 1 << 20;  // rows listed for the FP64 rescue kernel

int launch_point_wide(int type, graphgp_graph_t g, graphgp_factor_t f, const KernF& kf,
                      const RescueList& rl, const RowView& rv, cudaStream_t s) {
  const int64_t npts = rv.N - rv.n0;
  const size_t smem = kWideWarps * sizeof(WideWarp);
  const unsigned grid = grid_for((npts + kWideWarps - 1) / kWideWarps * 128, 128, 4);
#define GGP_PW(KT)                                                                           \
  GGP_CUDA(cudaFuncSetAttribute(point_factor_wide_kernel<KT>,                                \
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));    \
  point_factor_wide_kernel<KT><<<grid, 32 * kWideWarps, smem, s>>>(                          \
      g->xs, rv.nbr, rv.N, g->k, g->kp, rv.n0, kf, rv.b, f->sigma, f->logdet, f->not_pd, rl)
  switch (type) {
    case GRAPHGP_MATERN12: GGP_PW(GRAPHGP_MATERN12); break;
    case GRAPHGP_MATERN32: GGP_PW(GRAPHGP_MATERN32); break;
    case GRAPHGP_MATERN52: GGP_PW(GRAPHGP_MATERN52); break;
    default: GGP_PW(GRAPHGP_SQEXP); break;
  }
#undef GGP_PW
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

}  // namespace

int point_factor_rows(graphgp_graph_t g, graphgp_factor_t f, const KernF& kf, int type,
                      int64_t t0, int64_t t1, cudaStream_t s) {
  if (t1 <= t0) return GRAPHGP_OK;
  const int64_t npts = t1 - t0;
  const RowView rv{g->nbr + t0 * g->kp, f->b + t0 * g->kp, g->n0 + t1, g->n0 + t0};
  Scratch sc(s);
  RescueList rl;
  rl.cap = (unsigned long long)std::min<int64_t>(npts, kRescueListMax);
  GGP_TRY(sc.alloc(&rl.rows, rl.cap));
  GGP_TRY(sc.alloc(&rl.count, 1));
  GGP_CUDA(cudaMemsetAsync(rl.count, 0, sizeof(unsigned long long), s));
  switch (g->kp) {
    case 4: GGP_TRY(launch_point_pair<4>(type, g, f, kf, rl, rv, s)); return launch_rescue<4>(type, g, f, kf, rl, rv, s);
    case 8: GGP_TRY(launch_point_pair<8>(type, g, f, kf, rl, rv, s)); return launch_rescue<8>(type, g, f, kf, rl, rv, s);
    case 12: GGP_TRY(launch_point_pair<12>(type, g, f, kf, rl, rv, s)); return launch_rescue<12>(type, g, f, kf, rl, rv, s);
    case 16: GGP_TRY(launch_point_pair<16>(type, g, f, kf, rl, rv, s)); return launch_rescue<16>(type, g, f, kf, rl, rv, s);
    case 20:
    case 24: GGP_TRY(launch_point_oct<24>(type, g, f, kf, rl, rv, s)); return launch_rescue<24>(type, g, f, kf, rl, rv, s);
    case 28:
    case 32: GGP_TRY(launch_point_oct<32>(type, g, f, kf, rl, rv, s)); return launch_rescue<32>(type, g, f, kf, rl, rv, s);
    default: GGP_TRY(launch_point_wide(type, g, f, kf, rl, rv, s)); return launch_rescue<kWideK>(type, g, f, kf, rl, rv, s);
  }
}

int point_factor(graphgp_graph_t g, graphgp_factor_t f, const KernF& kf, int type,
                 cudaStream_t s) {
  return point_factor_rows(g, f, kf, type, 0, g->N - g->n0, s);
}

}  // namespace ggp

using namespace ggp;

static int factor_impl(graphgp_graph_t g, const graphgp_kernel* kern, int64_t p0, int64_t p1,
                       bool rows, void* stream, graphgp_factor_t* out) {
  if (!out) return GRAPHGP_ERR_INVALID;
  *out = nullptr;
  if (!g || !kern || kern->type < 0 || kern->type > 3 || !(kern->sigma2 > 0) ||
      !(kern->lengthscale > 0) || !(kern->nugget >= 0) || !std::isfinite(kern->rescue_tol))
    return GRAPHGP_ERR_INVALID;
  if (p0 < 0 || p1 > g->N || p0 > p1 || (p0 > 0 && p0 < g->n0) || (p0 == 0 && p1 < g->n0))
    return GRAPHGP_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  graphgp_factor_t f = new (std::nothrow) graphgp_factor_s();
  if (!f) return GRAPHGP_ERR_OOM;
  f->g = g;
  f->kern = *kern;
  if (rows) {
    f->row_begin = p0;
    f->row_end = p1;
  }
  auto fail = [&](int rc) {
    f->mem.free_all();
    delete f;
    return rc;
  };
  int rc = [&]() -> int {
    GGP_TRY(f->mem.alloc(&f->b, (g->N - g->n0) * g->kp));
    GGP_TRY(f->mem.alloc(&f->sigma, g->N));
    GGP_TRY(f->mem.alloc(&f->L0, (int64_t)g->n0 * g->n0));
    GGP_TRY(f->mem.alloc(&f->L0inv, (int64_t)g->n0 * g->n0));
    GGP_TRY(f->mem.alloc(&f->logdet, 1));
    GGP_TRY(f->mem.alloc(&f->not_pd, 1));
    GGP_CUDA(cudaMemsetAsync(f->logdet, 0, 8, s));
    GGP_CUDA(cudaMemsetAsync(f->not_pd, 0, 8, s));
    KernF kf = make_kernf(*kern, g);
    if (rows) {  // rows outside the range stay zero
      GGP_CUDA(cudaMemsetAsync(f->b, 0, (g->N - g->n0) * g->kp * sizeof(float), s));
      GGP_CUDA(cudaMemsetAsync(f->sigma, 0, g->N * sizeof(float), s));
      GGP_CUDA(cudaMemsetAsync(f->L0, 0, (int64_t)g->n0 * g->n0 * sizeof(float), s));
      GGP_CUDA(cudaMemsetAsync(f->L0inv, 0, (int64_t)g->n0 * g->n0 * sizeof(float), s));
    }
    if (p0 == 0) GGP_TRY(dense_factor(g, f, kf, kern->type, s));
    const int64_t t0 = std::max<int64_t>(p0, g->n0) - g->n0, t1 = std::max<int64_t>(p1 - g->n0, 0);
    GGP_TRY(point_factor_rows(g, f, kf, kern->type, t0, t1, s));
    return GRAPHGP_OK;
  }();
  if (rc < 0) return fail(rc);
  *out = f;
  return GRAPHGP_OK;
}

extern "C" int graphgp_factor(graphgp_graph_t g, const graphgp_kernel* kern, void* stream,
                              graphgp_factor_t* out) {
  if (!g) {
    if (out) *out = nullptr;
    return GRAPHGP_ERR_INVALID;
  }
  return factor_impl(g, kern, 0, g->N, false, stream, out);
}

extern "C" int graphgp_factor_rows(graphgp_graph_t g, const graphgp_kernel* kern,
                                   int64_t pos_begin, int64_t pos_end, void* stream,
                                   graphgp_factor_t* out) {
  if (!g) {
    if (out) *out = nullptr;
    return GRAPHGP_ERR_INVALID;
  }
  return factor_impl(g, kern, pos_begin, pos_end, true, stream, out);
}

extern "C" int graphgp_factor_export(graphgp_factor_t f, float* b_d, float* sigma_d, float* L0_d,
                                     void* stream) {
  if (!f) return GRAPHGP_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  graphgp_graph_t g = f->g;
  if (b_d && g->N > g->n0)
    GGP_CUDA(cudaMemcpy2DAsync(b_d, g->k * 4, f->b, g->kp * 4, g->k * 4, g->N - g->n0,
                               cudaMemcpyDeviceToDevice, s));
  if (sigma_d)
    GGP_CUDA(cudaMemcpyAsync(sigma_d, f->sigma, g->N * 4, cudaMemcpyDeviceToDevice, s));
  if (L0_d)
    GGP_CUDA(cudaMemcpyAsync(L0_d, f->L0, (int64_t)g->n0 * g->n0 * 4, cudaMemcpyDeviceToDevice, s));
  return GRAPHGP_OK;
}

extern "C" void graphgp_factor_destroy(graphgp_factor_t f) {
  if (!f) return;
  cudaDeviceSynchronize();
  f->mem.free_all();
  delete f;
}
