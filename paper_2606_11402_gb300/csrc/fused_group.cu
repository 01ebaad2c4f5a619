// On-the-fly sweeps (Alg. 1 as printed: the conditioning factor of every point
// recomputed inside the pass, nothing stored) for 16 < k <= 32: eight lanes per
// point, the factor and rescue decision of the factor kernel for these k
// (pointoct.cuh), so b and sigma are bit-identical to the stored factor's, and
// the dot b . v_c in the stored sweeps' summation order (oct_dot).
//
// generate: one cooperative launch over the depth levels with the level
// barrier of the stored sweep; a block factors its first points of a level
// before waiting at the barrier.  whiten: blocks stride over the positions,
// optionally reducing xi.xi and sum log sigma_i^2 in FP64.
#include "pointoct.cuh"

namespace ggp {
namespace {

__device__ inline void block_count(unsigned long long c, unsigned long long* out) {
  for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}

template <int K, int KT>
__global__ void __launch_bounds__(kPairThreads, OctLayout<K>::kBlocks) whiten_fused_group_kernel(
    const float4* __restrict__ xs, const int32_t* __restrict__ nbr, int64_t N, int k, int kp,
    int64_t n0, KernF kf, const float* __restrict__ v, float* __restrict__ xi,
    double* __restrict__ sq, double* __restrict__ logdet, unsigned long long* __restrict__ not_pd) {
  using OL = OctLayout<K>;
  extern __shared__ __align__(16) float psm[];
  const int lane = threadIdx.x & 31, r = lane & 7, first = (threadIdx.x >> 5) * 4;
  float* S = psm + (threadIdx.x >> 3) * OL::kStride;
  const uint64_t pol_v = l2_evict_last();
  LogAcc lacc;
  double local = 0.0;
  unsigned long long clamped = 0;
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
    float vv[K / 8];
    oct_gather<K, false>(vv, r, k, row, v, pol_v);
    oct_rescue<K, KT>(f, valid && oct_needs_rescue(f, kf), psm + first * OL::kStride, r, xs, row, k,
                      xq, kf);
    const float acc = oct_dot<K>(f.b, vv, S, r, kp);
    if (valid && r == 0) {
      const float out = (ld_keep_f(v + i, pol_v) - acc) / f.sigma;
      xi[i] = out;
      local += (double)out * (double)out;
      lacc.mul(f.sigma);
      clamped += f.clamped ? 1 : 0;
    }
  }
  if (sq) block_add_double(local, sq);
  if (logdet) block_add_double(lacc.log_value(), logdet);
  block_count(clamped, not_pd);
}

template <int K, int KT>
__global__ void __launch_bounds__(kPairThreads, OctLayout<K>::kBlocks) generate_fused_group_kernel(
    const float4* __restrict__ xs, const int32_t* __restrict__ nbr, int k, int kp, int64_t n0,
    KernF kf, const float* __restrict__ xi, float* v, const int64_t* __restrict__ level_off,
    int num_levels, LevelBarrier lb, unsigned long long* __restrict__ not_pd) {
  using OL = OctLayout<K>;
  __shared__ int s_flag;
  extern __shared__ __align__(16) float psm[];
  const int lane = threadIdx.x & 31, r = lane & 7, warp = threadIdx.x >> 5, first = warp * 4;
  float* S = psm + (threadIdx.x >> 3) * OL::kStride;
  const uint64_t pol_v = l2_evict_last();
  unsigned long long clamped = 0;
  for (int l = 1; l < num_levels; l++) {
    const int64_t lo = level_off[l], n = level_off[l + 1] - lo;
    const int64_t per = (n + gridDim.x - 1) / gridDim.x;
    const int64_t b0 = lo + min((int64_t)blockIdx.x * per, n);
    const int64_t hi = lo + min((int64_t)(blockIdx.x + 1) * per, n);
    const int64_t steps = (hi - b0 + OL::kPoints - 1) / OL::kPoints;
    if (steps == 0 && l > 1 && lb.wait(l - 1, gridDim.x, &s_flag)) return;
    for (int64_t st = 0; st < steps; st++) {
      // points dealt to the warps in turn: a warp recomputes its rows that need FP64
      // one after the other
      const int64_t q = b0 + st * OL::kPoints + (lane >> 3) * (kPairThreads / 32) + warp;
      const bool active = q < hi;
      const int64_t qq = active ? q : hi - 1;
      const int32_t* row = nbr + (qq - n0) * kp;
      const float4 xq = __ldg(xs + qq);
      oct_stage<K>(S, r, xs, row, kp);
      OctFactor<K> f;
      oct_factor<K, KT>(f, S, r, k, kf, xq);
      oct_rescue<K, KT>(f, active && oct_needs_rescue(f, kf), psm + first * OL::kStride, r, xs, row,
                        k, xq, kf);
      // the level's inputs are complete once every block arrived at l - 1
      if (st == 0 && l > 1 && lb.wait(l - 1, gridDim.x, &s_flag)) return;
      float vv[K / 8];
      oct_gather<K, true>(vv, r, k, row, v, pol_v);
      const float acc = oct_dot<K>(f.b, vv, S, r, kp);
      if (active && r == 0) {
        st_keep_f(v + q, fmaf(f.sigma, xi[q], acc), pol_v);
        clamped += f.clamped ? 1 : 0;
      }
    }
    __syncthreads();
    lb.arrive(l);
  }
  block_count(clamped, not_pd);
}

template <int K>
int whiten_group_kp(graphgp_graph_t g, int type, const KernF& kf, const float* v, float* xi,
                    double* sq, double* logdet, unsigned long long* not_pd, cudaStream_t s) {
  const int64_t npts = g->N - g->n0;
  if (npts <= 0) return GRAPHGP_OK;
  const unsigned grid = oct_grid<K>(npts);
  constexpr size_t smem = OctLayout<K>::kBytes;
#define GGP_WG(KT)                                                                          \
  GGP_CUDA(allow_dyn_smem(whiten_fused_group_kernel<K, KT>, smem));                         \
  whiten_fused_group_kernel<K, KT><<<grid, kPairThreads, smem, s>>>(                        \
      g->xs, g->nbr, g->N, g->k, g->kp, g->n0, kf, v, xi, sq, logdet, not_pd)
  switch (type) {
    case GRAPHGP_MATERN12: GGP_WG(GRAPHGP_MATERN12); break;
    case GRAPHGP_MATERN32: GGP_WG(GRAPHGP_MATERN32); break;
    case GRAPHGP_MATERN52: GGP_WG(GRAPHGP_MATERN52); break;
    default: GGP_WG(GRAPHGP_SQEXP); break;
  }
#undef GGP_WG
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

template <int K, int KT>
int generate_group_kt(graphgp_graph_t g, const KernF& kf, const float* xi, float* v,
                      unsigned long long* not_pd, cudaStream_t s) {
  constexpr size_t smem = OctLayout<K>::kBytes;
  GGP_CUDA(allow_dyn_smem(generate_fused_group_kernel<K, KT>, smem));
  static int max_grid_dev[kMaxDevices] = {};
  const int max_grid =
      coop_grid_cached(max_grid_dev, generate_fused_group_kernel<K, KT>, kPairThreads, smem);
  // Blocks for the largest level.  Where rows in FP64 are to be expected (no nugget,
  // or all of them asked for) one point per warp: the FP64 unit of an SM does two
  // lanes a clock, so what counts is the number of SMs.  Otherwise full blocks: more
  // of them only cost the barrier (30,011 points, k = 32: 2.67 ms with full blocks,
  // 2.73 / 2.99 / 3.65 with at least 152 / 304 / 456).
  const bool fp64 = kf.nugd == 0.0 || kf.resc_T < 0.0f;
  const int64_t per = fp64 ? kPairThreads / 32 : OctLayout<K>::kPoints;
  const int64_t want = (g->max_level_size + per - 1) / per;
  const int grid = (int)std::min<int64_t>(max_grid, std::max<int64_t>(want, 1));
  GGP_CUDA(cudaMemsetAsync(g->level_bar, 0, g->num_levels * sizeof(uint32_t), s));
  LevelBarrier lb{g->level_bar, g->err, g->max_spin};
  const float4* xs = g->xs;
  const int32_t* nbr = g->nbr;
  int k = g->k, kp = g->kp;
  int64_t n0 = g->n0;
  const int64_t* lo = g->level_off_d;
  int nl = g->num_levels;
  void* args[] = {(void*)&xs, (void*)&nbr, (void*)&k,  (void*)&kp, (void*)&n0, (void*)&kf,
                  (void*)&xi, (void*)&v,   (void*)&lo, (void*)&nl, (void*)&lb, (void*)&not_pd};
  GGP_CUDA(cudaLaunchCooperativeKernel((const void*)generate_fused_group_kernel<K, KT>,
                                       dim3(grid), dim3(kPairThreads), args, smem, s));
  return GRAPHGP_OK;
}

template <int K>
int generate_group_kp(graphgp_graph_t g, int type, const KernF& kf, const float* xi, float* v,
                      unsigned long long* not_pd, cudaStream_t s) {
  if (g->num_levels <= 1) return GRAPHGP_OK;
  switch (type) {
    case GRAPHGP_MATERN12: return generate_group_kt<K, GRAPHGP_MATERN12>(g, kf, xi, v, not_pd, s);
    case GRAPHGP_MATERN32: return generate_group_kt<K, GRAPHGP_MATERN32>(g, kf, xi, v, not_pd, s);
    case GRAPHGP_MATERN52: return generate_group_kt<K, GRAPHGP_MATERN52>(g, kf, xi, v, not_pd, s);
    default: return generate_group_kt<K, GRAPHGP_SQEXP>(g, kf, xi, v, not_pd, s);
  }
}

}  // namespace

// 16 < k <= 32 (row lengths 20, 24, 28, 32).
int whiten_fused_group(graphgp_graph_t g, int type, const KernF& kf, const float* v, float* xi,
                       double* sq, double* logdet, unsigned long long* not_pd, cudaStream_t s) {
  switch (g->kp) {
    case 20:
    case 24: return whiten_group_kp<24>(g, type, kf, v, xi, sq, logdet, not_pd, s);
    default: return whiten_group_kp<32>(g, type, kf, v, xi, sq, logdet, not_pd, s);
  }
}

int generate_fused_group(graphgp_graph_t g, int type, const KernF& kf, const float* xi, float* v,
                         unsigned long long* not_pd, cudaStream_t s) {
  switch (g->kp) {
    case 20:
    case 24: return generate_group_kp<24>(g, type, kf, xi, v, not_pd, s);
    default: return generate_group_kp<32>(g, type, kf, xi, v, not_pd, s);
  }
}

}  // namespace ggp
