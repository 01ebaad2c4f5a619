// Self-tests of the bounded device waits: a small launch waits for something that
// never happens -- the level barrier of the sweeps for more arrivals than there
// are blocks, the depth pass of the build (graph.cu) and the barrier-free sweep
// (sweeps.cu) for a value that nobody writes.  Each wait gives up after max_spin
// polls, records ERRBIT_TIMEOUT and returns, so the launch ends and the context
// stays usable; the host reads the error word.  And the root and reciprocal of the
// per-point factors on given arguments.
#include "pointpair.cuh"
#include "sweepsync.cuh"

namespace ggp {
namespace {

__global__ void barrier_timeout_kernel(LevelBarrier lb, uint32_t* reached) {
  __shared__ int s_flag;
  // nobody arrives at level 0, so gridDim.x + 1 arrivals never happen
  if (lb.wait(0, gridDim.x + 1, &s_flag)) return;
  if (threadIdx.x == 0) atomicAdd(reached, 1u);  // not reached while the bound works
}

// root[i] and inv[i] of x[i] by the scalar forms, pair[i] by the packed one whose
// other half is x[n - 1 - i].
__global__ void roots_kernel(const float* __restrict__ x, int64_t n, float* __restrict__ root,
                             float* __restrict__ pair, float* __restrict__ inv) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    root[i] = sqrt_newton(x[i]);
    const bool odd = i & 1;
    const float2 p = odd ? sqrt_pair(make_float2(x[n - 1 - i], x[i]))
                         : sqrt_pair(make_float2(x[i], x[n - 1 - i]));
    pair[i] = odd ? p.y : p.x;
    inv[i] = rcp_newton(x[i]);
  }
}

}  // namespace
}  // namespace ggp

using namespace ggp;

extern "C" int graphgp_selftest_wait(int which, int64_t max_spin, void* stream) {
  if (which < 0 || which > 2 || max_spin < 1 || max_spin > ((int64_t)1 << 30))
    return GRAPHGP_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  Scratch sc(s);
  uint32_t* words = nullptr;  // [0] count, [1] error word, [2] reached
  GGP_TRY(sc.alloc(&words, 4));
  GGP_CUDA(cudaMemsetAsync(words, 0, 4 * sizeof(uint32_t), s));
  if (which == 0) {
    LevelBarrier lb{words, words + 1, max_spin};
    uint32_t* reached = words + 2;
    void* args[] = {(void*)&lb, (void*)&reached};
    GGP_CUDA(cudaLaunchCooperativeKernel((const void*)barrier_timeout_kernel, dim3(2), dim3(64),
                                         args, 0, s));
  } else if (which == 1) {
    GGP_TRY(depth_wait_selftest(max_spin, words + 1, s));
  } else {
    GGP_TRY(flow_wait_selftest(max_spin, words + 1, s));
  }
  uint32_t h[4] = {0, 0, 0, 0};
  GGP_CUDA(cudaMemcpyAsync(h, words, sizeof(h), cudaMemcpyDeviceToHost, s));
  GGP_CUDA(cudaStreamSynchronize(s));
  if (h[2] != 0) return GRAPHGP_ERR_INVALID;  // a wait passed without arrivals
  return (h[1] & ERRBIT_TIMEOUT) ? GRAPHGP_ERR_TIMEOUT : GRAPHGP_OK;
}

extern "C" int graphgp_selftest_wait_timeout(int64_t max_spin, void* stream) {
  return graphgp_selftest_wait(0, max_spin, stream);
}

extern "C" int graphgp_selftest_roots(const float* x_d, int64_t n, float* root_d, float* pair_d,
                                      float* inv_d, void* stream) {
  if (!x_d || n < 1 || !root_d || !pair_d || !inv_d) return GRAPHGP_ERR_INVALID;
  roots_kernel<<<grid_for(n, 256), 256, 0, (cudaStream_t)stream>>>(x_d, n, root_d, pair_d, inv_d);
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

// Target of the device code actually loaded: binaryVersion of one of the
// library's kernels (major * 10 + minor, 103 for sm_103a).
extern "C" int graphgp_binary_version(int* version) {
  if (!version) return GRAPHGP_ERR_INVALID;
  cudaFuncAttributes a;
  GGP_CUDA(cudaFuncGetAttributes(&a, (const void*)barrier_timeout_kernel));
  *version = a.binaryVersion;
  return GRAPHGP_OK;
}
