// Level sweeps of Alg. 1 (generate, v = L xi) and the inverse application
// and log-determinant of Sec. 3 (whiten, xi = L^-1 v; logdet; NLL).
//
// generate: v_0 = L0 xi_0 for the dense block, then batch by batch
// (Sec. 2.2: points of one depth level are conditionally independent)
// v_i = b_i . v_c(i) + sigma_i xi_i; every neighbour lies in an earlier level.
// One cooperative launch walks the levels with a grid-wide barrier between
// consecutive levels (sweepsync.cuh).  Rows, sigma and xi do not depend on
// the field: each lane group loads those of its next step before gathering
// the current one, and those of a level's first step before the barrier, so
// the row stream overlaps both the gathers and the barrier.  The depth levels
// at both ends of the sweep hold a few dozen to a few hundred points (about
// 90 levels at any N); each of those runs is done by a single block that
// synchronises with __syncthreads, since a grid barrier per level costs
// more than the level's work there: the first run with its field in shared
// memory, the last with gathers from L2.  Clouds of at most kFlowEntries row
// entries (and kFlowLevel a level) have no barrier after the first run: a gathered
// value is its own flag.
//
// whiten: xi_i = (v_i - b_i . v_c(i)) / sigma_i has no dependencies.  Blocks
// walk spatial tiles through every level (plus xi_0 = L0^-1 v_0 for the
// dense block), so the gathered v lines of a tile stay in L1; rows are
// streamed without L1 allocation, v is kept in L2 (evict-last).  With fewer
// than four tiles per SM the positions are taken in order by all blocks.
#include <algorithm>

#include "sweepsync.cuh"

namespace ggp {
namespace {

// y[i] = sum_{m <= i} M[i][m] x[m] for the n0 x n0 lower-triangular M; one
// warp per row.  Optionally accumulates sum y_i^2 in FP64.
__global__ void dense_lower_matvec_kernel(const float* __restrict__ M, const float* __restrict__ x,
                                          float* __restrict__ y, int n0, double* __restrict__ sq) {
  int warps = (gridDim.x * blockDim.x) >> 5;
  int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int lane = threadIdx.x & 31;
  for (int i = w; i < n0; i += warps) {
    const float* r = M + (int64_t)i * n0;
    float s = 0.0f;
    for (int m = lane; m <= i; m += 32) s = fmaf(r[m], x[m], s);
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      y[i] = s;
      if (sq) atomicAdd(sq, (double)s * (double)s);
    }
  }
}

template <int KP>
struct Row {
  int4 n[KP / 4];
  float4 w[KP / 4];
};

template <int KP>
__device__ __forceinline__ void load_row(Row<KP>& r, const int32_t* __restrict__ nbr,
                                         const float* __restrict__ b, int64_t row, uint64_t pol) {
  const int4* np = reinterpret_cast<const int4*>(nbr + row * KP);
  const float4* bp = reinterpret_cast<const float4*>(b + row * KP);
#pragma unroll
  for (int q = 0; q < KP / 4; q++) {
    r.n[q] = ld_stream_i4(np + q, pol);
    r.w[q] = ld_stream_f4(bp + q, pol);
  }
}


// The same row, loaded without allocating in L1 (the whiten sweep keeps L1
// for the gathered field values of its tile).
template <int KP>
__device__ __forceinline__ void load_row_na(Row<KP>& r, const int32_t* __restrict__ nbr,
                                            const float* __restrict__ b, int64_t row,
                                            uint64_t pol) {
  const int4* np = reinterpret_cast<const int4*>(nbr + row * KP);
  const float4* bp = reinterpret_cast<const float4*>(b + row * KP);
#pragma unroll
  for (int q = 0; q < KP / 4; q++) {
    r.n[q] = ld_stream_na_i4(np + q, pol);
    r.w[q] = ld_stream_na_f4(bp + q, pol);
  }
}

// sum_a b_a v[c_a].  LEVEL: v is written level by level in the same launch;
// the gathered entries belong to earlier levels, published by the barrier.
template <int KP, bool LEVEL>
__device__ __forceinline__ float gather_dot(const Row<KP>& r, const float* __restrict__ v,
                                            uint64_t pol) {
  float acc0 = 0.0f, acc1 = 0.0f;
#pragma unroll
  for (int q = 0; q < KP / 4; q++) {
    float v0, v1, v2, v3;
    if (LEVEL) {
      v0 = ld_level_f(v + r.n[q].x, pol); v1 = ld_level_f(v + r.n[q].y, pol);
      v2 = ld_level_f(v + r.n[q].z, pol); v3 = ld_level_f(v + r.n[q].w, pol);
    } else {
      v0 = ld_keep_f(v + r.n[q].x, pol); v1 = ld_keep_f(v + r.n[q].y, pol);
      v2 = ld_keep_f(v + r.n[q].z, pol); v3 = ld_keep_f(v + r.n[q].w, pol);
    }
    acc0 = fmaf(r.w[q].x, v0, acc0);
    acc1 = fmaf(r.w[q].y, v1, acc1);
    acc0 = fmaf(r.w[q].z, v2, acc0);
    acc1 = fmaf(r.w[q].w, v3, acc1);
  }
  return acc0 + acc1;
}

constexpr int kSweepThreads = 256;


// Positions per lane group and step of generate_kernel: as many as keep the
// two row buffers below about 64 registers.
__host__ __device__ constexpr int gen_steps(int hp) { return hp <= 4 ? 4 : (hp <= 8 ? 2 : 1); }

// Levels [l_first, l_end) of generate.  LANES threads share one position:
// lane h holds entries [h HP, (h+1) HP) of the row (HP = KP / LANES) and the
// partial sums meet in shuffles.  A lane group takes U positions per step,
// and the rows, sigma and xi of its next step are loaded before the gathers
// of the current one, so their DRAM latency hides under the gathers.  The
// first step of a level is loaded before the level's wait (rows do not depend
// on the field).
//   GRID: a cooperative launch; block b takes the b-th of gridDim.x equal
//         slices of every level and waits at the grid-wide level barrier.
//   !GRID: one block takes whole levels and waits at __syncthreads (levels
//         of a few hundred points, where the grid barrier would dominate).
template <int KP, int LANES, int U, int NT, bool GRID>
__device__ __forceinline__ void gen_levels(const int32_t* __restrict__ nbr,
                                           const float* __restrict__ b,
                                           const float* __restrict__ sigma,
                                           const float* __restrict__ xi, float* v,
                                           const int64_t* __restrict__ level_off, int l_first,
                                           int l_end, int64_t n0, const LevelBarrier& lb,
                                           int* s_flag) {
  constexpr int HP = KP / LANES;   // row entries per lane
  constexpr int GPB = NT / LANES;  // lane groups per block
  constexpr int PPB = U * GPB;     // positions per block step
  const uint64_t pol_rows = l2_evict_first();
  const uint64_t pol_v = l2_evict_last();
  const int h = threadIdx.x % LANES;
  const int slot = threadIdx.x / LANES;
  const int32_t* nb = nbr + h * HP;
  const float* bw = b + h * HP;
  Row<HP> rn[U];
  float sgn[U], xn[U];
  for (int l = l_first; l < l_end; l++) {
    const int64_t lo = level_off[l], n = level_off[l + 1] - lo;
    int64_t b0 = lo, hi = lo + n;
    if (GRID) {
      const int64_t per = (n + gridDim.x - 1) / gridDim.x;
      b0 = lo + min((int64_t)blockIdx.x * per, n);
      hi = lo + min((int64_t)(blockIdx.x + 1) * per, n);
    }
    int64_t p = b0 + slot;
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int64_t q = p + u * GPB;
      sgn[u] = xn[u] = 0.0f;
      if (q < hi) {
        load_row<HP>(rn[u], nb, bw, (q - n0) * LANES, pol_rows);
        if (h == 0) {
          sgn[u] = ld_stream_f(sigma + q, pol_rows);
          xn[u] = ld_stream_f(xi + q, pol_rows);
        }
      }
    }
    if (l > l_first) {
      if (GRID) {
        if (lb.wait(l - 1, gridDim.x, s_flag)) return;
      } else {
        __syncthreads();
      }
    }
    const int64_t steps = (hi - b0 + PPB - 1) / PPB;
    for (int64_t st = 0; st < steps; st++) {
      Row<HP> r[U];
      float sg[U], x[U];
#pragma unroll
      for (int u = 0; u < U; u++) {
        r[u] = rn[u];
        sg[u] = sgn[u];
        x[u] = xn[u];
      }
      const int64_t pn = p + PPB;
#pragma unroll
      for (int u = 0; u < U; u++) {
        const int64_t qn = pn + u * GPB;
        if (qn < hi) {
          load_row<HP>(rn[u], nb, bw, (qn - n0) * LANES, pol_rows);
          if (h == 0) {
            sgn[u] = ld_stream_f(sigma + qn, pol_rows);
            xn[u] = ld_stream_f(xi + qn, pol_rows);
          }
        }
      }
      float acc[U];
#pragma unroll
      for (int u = 0; u < U; u++) {
        const int64_t q = p + u * GPB;
        acc[u] = q < hi ? gather_dot<HP, true>(r[u], v, pol_v) : 0.0f;
      }
#pragma unroll
      for (int u = 0; u < U; u++) {
        if (LANES >= 4) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], 2);
        if (LANES >= 2) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], 1);
        const int64_t q = p + u * GPB;
        if (q < hi && h == 0) st_keep_f(v + q, fmaf(sg[u], x[u], acc[u]), pol_v);
      }
      p = pn;
    }
    if (GRID) {
      __syncthreads();
      lb.arrive(l);
    }
  }
}

template <int KP, int LANES, int U>
__global__ void __launch_bounds__(kSweepThreads) generate_kernel(
    const int32_t* __restrict__ nbr, const float* __restrict__ b, const float* __restrict__ sigma,
    const float* __restrict__ xi, float* v, const int64_t* __restrict__ level_off, int l_first,
    int l_end, int64_t n0, LevelBarrier lb) {
  __shared__ int s_flag;
  gen_levels<KP, LANES, U, kSweepThreads, true>(nbr, b, sigma, xi, v, level_off, l_first, l_end,
                                                n0, lb, &s_flag);
}

// One block of small_threads(KP) threads for runs of small levels.
__host__ __device__ constexpr int small_threads(int hp) { return hp <= 4 ? 1024 : (hp <= 8 ? 512 : 256); }
__host__ __device__ constexpr int small_steps(int hp) { return hp <= 8 ? 2 : 1; }

template <int KP, int LANES>
__global__ void __launch_bounds__(small_threads(KP / LANES), 1) generate_small_kernel(
    const int32_t* __restrict__ nbr, const float* __restrict__ b, const float* __restrict__ sigma,
    const float* __restrict__ xi, float* v, const int64_t* __restrict__ level_off, int l_first,
    int l_end, int64_t n0) {
  constexpr int HP = KP / LANES;
  LevelBarrier none{nullptr, nullptr, 0};
  gen_levels<KP, LANES, small_steps(HP), small_threads(HP), false>(
      nbr, b, sigma, xi, v, level_off, l_first, l_end, n0, none, nullptr);
}

// ---- the first levels of generate in one block ------------------------------------
// The levels up to the first large one hold a few dozen to a few hundred points
// each, and their neighbours are all among the first few ten thousand positions:
// one block keeps that part of the field in shared memory, so a level costs a
// block barrier and a shared-memory gather instead of a round trip through L2.
// Row slices, sigma and xi are loaded D steps ahead, across level boundaries.
// Bound by the chain barrier - gather - shuffle - store of each level.
// generate against one block that gathers from L2 and a grid barrier for every
// level above kTail: 46.4 -> 29.7 us (4096 points, k = 8), 66.9 -> 39.1 (4096,
// k = 16), 88.4 -> 59.2 (10007, k = 16), 220 -> 188 (127001, k = 16).
// Row slices of 28 entries (k = 25 .. 28, one lane per position) have half the
// threads: two buffers of them need 112 registers.
__host__ __device__ constexpr int head_threads(int hp) { return hp > 20 ? 256 : 512; }
constexpr int64_t kHeadPoints = 49152;  // positions held (192 KB)
constexpr int kHeadLevels = 4096;
__host__ __device__ constexpr int head_depth(int hp) { return hp <= 4 ? 3 : (hp <= 8 ? 2 : 1); }

template <int KP, int LANES>
__global__ void __launch_bounds__(head_threads(KP / LANES), 1) generate_head_kernel(
    const int32_t* __restrict__ nbr, const float* __restrict__ b, const float* __restrict__ sigma,
    const float* __restrict__ xi, float* __restrict__ v, const int64_t* __restrict__ level_off,
    int l_end, int64_t n0) {
  constexpr int HP = KP / LANES, NT = head_threads(HP), PPB = NT / LANES, D = head_depth(HP);
  extern __shared__ float s_v[];  // the field up to the last level's end, then the offsets
  const int32_t end = (int32_t)level_off[l_end];
  int32_t* s_lo = reinterpret_cast<int32_t*>(s_v + end);
  for (int l = threadIdx.x; l <= l_end; l += NT) s_lo[l] = (int32_t)level_off[l];
  for (int i = threadIdx.x; i < (int)n0; i += NT) s_v[i] = v[i];
  __syncthreads();
  const int h = threadIdx.x % LANES, slot = threadIdx.x / LANES;
  const uint64_t pol = l2_policy<0>();
  const int32_t* nb = nbr + h * HP;
  const float* bw = b + h * HP;
  Row<HP> r[D + 1];
  float sg[D + 1], x[D + 1];
  // step: level l, first position p; load into buffer i
  int ll = 1, lp = s_lo[1];  // the next step to load
  auto load = [&](Row<HP>& row, float& s, float& xv) {
    if (ll >= l_end) return;
    const int q = lp + slot;
    s = xv = 0.0f;
    if (q < s_lo[ll + 1]) {
      load_row<HP>(row, nb, bw, ((int64_t)q - n0) * LANES, pol);
      if (h == 0) {
        s = ld_stream_f(sigma + q, pol);
        xv = ld_stream_f(xi + q, pol);
      }
    }
    lp += PPB;
    if (lp >= s_lo[ll + 1]) lp = s_lo[++ll];
  };
#pragma unroll
  for (int i = 0; i < D; i++) load(r[i], sg[i], x[i]);
  int l = 1, p = s_lo[1];
  while (l < l_end) {
#pragma unroll
    for (int i = 0; i <= D; i++) {  // buffer i holds this step, i + D is refilled
      if (l >= l_end) break;
      load(r[(i + D) % (D + 1)], sg[(i + D) % (D + 1)], x[(i + D) % (D + 1)]);
      if (p == s_lo[l]) __syncthreads();  // the levels before are complete
      const int q = p + slot;
      const bool act = q < s_lo[l + 1];
      float a0 = 0.0f, a1 = 0.0f;  // gather_dot's order
      if (act) {
#pragma unroll
        for (int c = 0; c < HP / 4; c++) {
          a0 = fmaf(r[i].w[c].x, s_v[r[i].n[c].x], a0);
          a1 = fmaf(r[i].w[c].y, s_v[r[i].n[c].y], a1);
          a0 = fmaf(r[i].w[c].z, s_v[r[i].n[c].z], a0);
          a1 = fmaf(r[i].w[c].w, s_v[r[i].n[c].w], a1);
        }
      }
      float acc = a0 + a1;
      if (LANES >= 4) acc += __shfl_xor_sync(0xffffffffu, acc, 2);
      if (LANES >= 2) acc += __shfl_xor_sync(0xffffffffu, acc, 1);
      if (act && h == 0) {
        const float out = fmaf(sg[i], x[i], acc);
        s_v[q] = out;
        v[q] = out;
      }
      p += PPB;
      if (p >= s_lo[l + 1]) p = s_lo[++l];
    }
  }
}

// ---- generate by dataflow ------------------------------------------------------
// Small and medium clouds: no barrier between levels.  v starts as the all-ones
// NaN (0xffffffff; a NaN result of the arithmetic is the canonical 0x7fffffff,
// and a store maps the one to the other all the same), and a gathered entry that
// still holds it is read again at L2 until its value is there: the value is its own flag, so
// a level costs one trip through L2 instead of a barrier and a gather behind it.
// Every warp takes its own slice of each level (slices of consecutive warps lie
// on different SMs, so a level of a few hundred points is spread over as many),
// in level order and without waiting for the other warps of its block, and
// loads the rows of its next step, of whichever level, before it gathers the
// current one.  A cooperative launch: all warps are resident, and the lowest
// unfinished level never waits for a later one.  Waits are bounded as in the
// level barrier (a warp may wait here for many levels, so it gets kFlowPolls
// polls more for each).  Large levels gather most values from L1 behind the
// barrier, which a flag read at L2 cannot, so they keep the barrier
// (launch_generate has the line and both sides).
constexpr uint32_t kNotYet = 0xffffffffu;
constexpr int kFlowMaxLevels = 4096;  // level table in shared memory
constexpr int64_t kFlowEntries = 8 << 20;  // N times the padded row length
constexpr int64_t kFlowLevel = 256 << 10;
constexpr int64_t kFlowPolls = 1024;

__device__ __forceinline__ uint32_t ld_flag(const float* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_flag(float* p, float v) {
  uint32_t u = __float_as_uint(v);
  if (u == kNotYet) u = 0x7fffffffu;
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(u) : "memory");
}

template <int KP, int LANES, int U>
__global__ void __launch_bounds__(kSweepThreads) generate_flow_kernel(
    const int32_t* __restrict__ nbr, const float* __restrict__ b, const float* __restrict__ sigma,
    const float* __restrict__ xi, float* v, const int64_t* __restrict__ level_off, int l_first,
    int num_levels, int64_t n0, int64_t max_spin, uint32_t* err) {
  constexpr int HP = KP / LANES, PPW = 32 / LANES;  // row entries per lane, positions per warp
  extern __shared__ int32_t s_lo[];                 // [num_levels + 1], then slice lengths
  int32_t* s_per = s_lo + num_levels + 1;
  const int warps = gridDim.x * (kSweepThreads / 32);
  for (int l = threadIdx.x; l <= num_levels; l += kSweepThreads) s_lo[l] = (int32_t)level_off[l];
  __syncthreads();
  for (int l = threadIdx.x; l < num_levels; l += kSweepThreads) {
    const uint32_t n = (uint32_t)(s_lo[l + 1] - s_lo[l]);
    const uint32_t per = (n + warps - 1) / warps;
    s_per[l] = (int32_t)((per + PPW - 1) / PPW * PPW);
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, h = lane % LANES, grp = lane / LANES;
  const int w = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const uint64_t pol = l2_policy<0>();
  const int32_t* nb = nbr + h * HP;
  const float* bw = b + h * HP;
  struct Step {
    int l;
    int64_t p, end;
  };
  auto first_of = [&](int l) {  // the warp's first step in level l or later
    for (; l < num_levels; l++) {
      const int64_t off = (int64_t)w * s_per[l];
      const int64_t n = s_lo[l + 1] - s_lo[l];
      if (off < n) return Step{l, s_lo[l] + off, s_lo[l] + min(off + s_per[l], n)};
    }
    return Step{l, 0, 0};
  };
  Row<HP> rn[U];
  float sgn[U], xn[U];
  auto load = [&](const Step& st) {
#pragma unroll
    for (int u = 0; u < U; u++) {
      const int64_t q = st.p + u * PPW + grp;
      sgn[u] = xn[u] = 0.0f;
      if (q < st.end) {
        load_row<HP>(rn[u], nb, bw, (q - n0) * LANES, pol);
        if (h == 0) {
          sgn[u] = ld_stream_f(sigma + q, pol);
          xn[u] = ld_stream_f(xi + q, pol);
        }
      }
    }
  };
  Step cur = first_of(l_first);
  if (cur.l >= num_levels) return;
  load(cur);
  while (true) {
    Row<HP> r[U];
    float sg[U], x[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
      r[u] = rn[u];
      sg[u] = sgn[u];
      x[u] = xn[u];
    }
    Step nxt = cur;
    nxt.p += U * PPW;
    if (nxt.p >= nxt.end) nxt = first_of(cur.l + 1);
    const bool more = nxt.l < num_levels;
    if (more) load(nxt);
    float acc[U];
    bool dead = false;
#pragma unroll
    for (int u = 0; u < U; u++) {
      acc[u] = 0.0f;
      if (cur.p + u * PPW + grp < cur.end) {
        uint32_t g[HP];
#pragma unroll
        for (int q = 0; q < HP / 4; q++) {
          g[4 * q] = ld_flag(v + r[u].n[q].x);
          g[4 * q + 1] = ld_flag(v + r[u].n[q].y);
          g[4 * q + 2] = ld_flag(v + r[u].n[q].z);
          g[4 * q + 3] = ld_flag(v + r[u].n[q].w);
        }
        int64_t spins = 0;
        while (true) {
          bool wait = false;
#pragma unroll
          for (int q = 0; q < HP; q++) wait |= g[q] == kNotYet;
          if (!wait || dead) break;
#pragma unroll
          for (int q = 0; q < HP / 4; q++) {
            if (g[4 * q] == kNotYet) g[4 * q] = ld_flag(v + r[u].n[q].x);
            if (g[4 * q + 1] == kNotYet) g[4 * q + 1] = ld_flag(v + r[u].n[q].y);
            if (g[4 * q + 2] == kNotYet) g[4 * q + 2] = ld_flag(v + r[u].n[q].z);
            if (g[4 * q + 3] == kNotYet) g[4 * q + 3] = ld_flag(v + r[u].n[q].w);
          }
          __nanosleep(20);
          if ((++spins & 63) == 0) {
            if (spins > max_spin) atomicOr(err, ERRBIT_TIMEOUT);
            dead = sync_ld_acquire(err) & ERRBIT_TIMEOUT;
          }
        }
        float a0 = 0.0f, a1 = 0.0f;  // gather_dot's order
#pragma unroll
        for (int q = 0; q < HP / 4; q++) {
          a0 = fmaf(r[u].w[q].x, __uint_as_float(g[4 * q]), a0);
          a1 = fmaf(r[u].w[q].y, __uint_as_float(g[4 * q + 1]), a1);
          a0 = fmaf(r[u].w[q].z, __uint_as_float(g[4 * q + 2]), a0);
          a1 = fmaf(r[u].w[q].w, __uint_as_float(g[4 * q + 3]), a1);
        }
        acc[u] = a0 + a1;
      }
    }
    if (__any_sync(0xffffffffu, dead)) return;
#pragma unroll
    for (int u = 0; u < U; u++) {
      if (LANES >= 4) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], 2);
      if (LANES >= 2) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], 1);
      const int64_t q = cur.p + u * PPW + grp;
      if (q < cur.end && h == 0) st_flag(v + q, fmaf(sg[u], x[u], acc[u]));
    }
    if (!more) return;
    cur = nxt;
  }
}

template <int KP>
int launch_generate_flow(graphgp_graph_t g, graphgp_factor_t f, const float* xi, float* v,
                         int l_first, cudaStream_t s) {
  constexpr int LANES = gen_lanes(KP), HP = KP / LANES, U = HP <= 4 ? 2 : 1;
  int L = g->num_levels;
  int64_t n0 = g->n0, spin = g->max_spin + kFlowPolls * L;
  const int64_t p0 = g->level_off_h[l_first];
  GGP_CUDA(cudaMemsetAsync(v + p0, 0xff, (g->N - p0) * sizeof(float), s));
  auto kern = generate_flow_kernel<KP, LANES, U>;
  const size_t smem = (2 * (size_t)L + 1) * sizeof(int32_t);
  static int max_grid_dev[kMaxDevices] = {};
  const int max_grid = coop_grid_cached(max_grid_dev, kern, kSweepThreads,
                                        (2 * (size_t)kFlowMaxLevels + 1) * sizeof(int32_t));
  // one position per lane group of the largest level is as wide as it gets
  const int64_t want = (g->max_level_size * LANES + kSweepThreads - 1) / kSweepThreads;
  const int grid = (int)std::min<int64_t>(max_grid, std::max<int64_t>(want, 1));
  const int32_t* nbr = g->nbr;
  const float *bw = f->b, *sg = f->sigma;
  const int64_t* lod = g->level_off_d;
  uint32_t* err = g->err;
  void* args[] = {(void*)&nbr, (void*)&bw, (void*)&sg, (void*)&xi,   (void*)&v,
                  (void*)&lod, (void*)&l_first, (void*)&L, (void*)&n0, (void*)&spin, (void*)&err};
  GGP_CUDA(cudaLaunchCooperativeKernel((const void*)kern, dim3(grid), dim3(kSweepThreads), args,
                                       smem, s));
  return GRAPHGP_OK;
}

// whiten in position order, LANES lanes per position and U positions per lane
// group and step.  Bound by DRAM once the rows exceed L2 (10^6 points, k = 16:
// 140 MB in 60 us) and by latency below.
template <int KP, int LANES, int U>
__global__ void __launch_bounds__(256) whiten_flat_kernel(
    const int32_t* __restrict__ nbr, const float* __restrict__ b, const float* __restrict__ sigma,
    const float* __restrict__ v, float* __restrict__ xi, int64_t N, int64_t n0,
    double* __restrict__ sq) {
  constexpr int HP = KP / LANES, GPB = 256 / LANES;
  const uint64_t pol_rows = l2_policy<0>();
  const uint64_t pol_v = l2_evict_last();
  const int h = threadIdx.x % LANES;
  double local = 0.0;
  for (int64_t p0 = n0 + (int64_t)blockIdx.x * (GPB * U) + threadIdx.x / LANES;
       p0 - threadIdx.x / LANES < N; p0 += (int64_t)gridDim.x * (GPB * U)) {
    Row<HP> r[U];
    float acc[U];
#pragma unroll
    for (int u = 0; u < U; u++)
      if (p0 + u * GPB < N)
        load_row_na<HP>(r[u], nbr + h * HP, b + h * HP, (p0 + u * GPB - n0) * LANES, pol_rows);
#pragma unroll
    for (int u = 0; u < U; u++)
      acc[u] = p0 + u * GPB < N ? gather_dot<HP, false>(r[u], v, pol_v) : 0.0f;
#pragma unroll
    for (int u = 0; u < U; u++) {
      if (LANES >= 4) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], 2);
      if (LANES >= 2) acc[u] += __shfl_xor_sync(0xffffffffu, acc[u], 1);
      const int64_t pos = p0 + u * GPB;
      if (pos < N && h == 0) {
        const float out = (ld_keep_f(v + pos, pol_v) - acc[u]) / ld_stream_na_f(sigma + pos, pol_rows);
        st_stream_f(xi + pos, out, pol_rows);
        if (sq) local += (double)out * (double)out;
      }
    }
  }
  if (sq) {
    __shared__ double red[8];
    for (int o = 16; o; o >>= 1) local += __shfl_xor_sync(0xffffffffu, local, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = local;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int i = 0; i < (int)(blockDim.x >> 5); i++) s += red[i];
      atomicAdd(sq, s);
    }
  }
}

// whiten over spatial tiles: a block takes one tile (a k-d in-order rank range
// of kTileR points) and walks its positions in every level >= 1.  The gathers
// of a tile land mostly on the same tile's v values, which stay in L1.
template <int KP>
__global__ void __launch_bounds__(256) whiten_tiles_kernel(
    const int32_t* __restrict__ nbr, const float* __restrict__ b, const float* __restrict__ sigma,
    const float* __restrict__ v, float* __restrict__ xi, int64_t n0,
    const int32_t* __restrict__ tile_start, int64_t n_tiles, int num_levels,
    double* __restrict__ sq) {
  extern __shared__ int32_t sm[];
  int32_t* s_start = sm;               // [num_levels]
  int32_t* s_pref = sm + num_levels;   // [num_levels + 1]
  __shared__ int32_t s_carry;
  const uint64_t pol_rows = l2_policy<0>();  // whiten: rows evict-normal (measured best)
  const uint64_t pol_v = l2_evict_last();
  double local = 0.0;
  for (int64_t t = blockIdx.x; t < n_tiles; t += gridDim.x) {
    const int32_t* ts = tile_start + t * num_levels;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    // exclusive prefix of the tile's counts over levels 1..L-1 (level 0 is dense)
    for (int base = 1; base < num_levels; base += blockDim.x) {
      int l = base + threadIdx.x;
      int32_t c = 0;
      if (l < num_levels) {
        int32_t a0 = ts[l];
        c = ts[num_levels + l] - a0;
        s_start[l] = a0;
      }
      // block-wide inclusive scan of c
      int32_t x = c;
      for (int o = 1; o < 32; o <<= 1) {
        int32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if ((threadIdx.x & 31) >= o) x += y;
      }
      __shared__ int32_t wsum[8];
      if ((threadIdx.x & 31) == 31) wsum[threadIdx.x >> 5] = x;
      __syncthreads();
      int32_t wpre = 0;
      for (int w = 0; w < (int)(threadIdx.x >> 5); w++) wpre += wsum[w];
      int32_t carry = s_carry;
      if (l < num_levels) s_pref[l] = carry + wpre + x - c;
      __syncthreads();
      if (threadIdx.x == blockDim.x - 1) s_carry = carry + wpre + x;
      __syncthreads();
    }
    const int32_t total = s_carry;
    // LANES lanes share a position; lane h holds row entries [h HP, (h+1) HP),
    // so a warp reads 32/LANES consecutive rows as whole sectors
    constexpr int LANES = gen_lanes(KP), HP = KP / LANES, GPB = 256 / LANES;
    const int h = threadIdx.x % LANES;
    const int32_t steps = (total + GPB - 1) / GPB;
    for (int32_t st = 0; st < steps; st++) {
      const int32_t vi = st * GPB + (int32_t)threadIdx.x / LANES;
      const bool act = vi < total;
      int64_t pos = 0;
      float acc = 0.0f;
      if (act) {
        // level of vi: last l >= 1 with s_pref[l] <= vi
        int lo = 1, hi = num_levels - 1;
        while (lo < hi) {
          int mid = (lo + hi + 1) >> 1;
          if (s_pref[mid] <= vi) lo = mid; else hi = mid - 1;
        }
        pos = (int64_t)s_start[lo] + (vi - s_pref[lo]);
        Row<HP> r;
        load_row_na<HP>(r, nbr + h * HP, b + h * HP, (pos - n0) * LANES, pol_rows);
        acc = gather_dot<HP, false>(r, v, pol_v);
      }
      if (LANES >= 4) acc += __shfl_xor_sync(0xffffffffu, acc, 2);
      if (LANES >= 2) acc += __shfl_xor_sync(0xffffffffu, acc, 1);
      if (act && h == 0) {
        float sg = ld_stream_na_f(sigma + pos, pol_rows);
        float vv = ld_keep_f(v + pos, pol_v);
        float out = (vv - acc) / sg;
        st_stream_f(xi + pos, out, pol_rows);
        if (sq) local += (double)out * (double)out;
      }
    }
    __syncthreads();
  }
  if (sq) {
    __shared__ double red[8];
    for (int o = 16; o; o >>= 1) local += __shfl_xor_sync(0xffffffffu, local, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = local;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int i = 0; i < (int)(blockDim.x >> 5); i++) s += red[i];
      atomicAdd(sq, s);
    }
  }
}

__global__ void nll_finish_kernel(const double* __restrict__ sq, const double* __restrict__ logdet,
                                  double* __restrict__ out) {
  out[0] = 0.5 * sq[0] + 0.5 * logdet[0];
}

template <int KP>
int launch_generate(graphgp_graph_t g, graphgp_factor_t f, const float* xi, float* v,
                    cudaStream_t s) {
  const int L = g->num_levels;
  if (L <= 1) return GRAPHGP_OK;
  constexpr int LANES = gen_lanes(KP), HP = KP / LANES, U = gen_steps(HP);
  // The run of small levels that the sweep starts with goes to one block with its
  // field in shared memory: levels of at most kSmall points and kSmallEntries row
  // entries, which bound the block's loads.  generate with the line at 4 / 8 / 16 /
  // 64 Ki entries, us: 30011 points, k = 16: 86 / 90 / 105 / 105, k = 32: 151 / 152 /
  // 170 / 194, k = 64: 364 / 338 / 387 / 455; 127001, k = 16: 135 / 133 / 144 / 144,
  // k = 48: 425 / 380 / 368 / 495; 10^6, k = 8: 132 / 129 / 130 / 130.  One lane per
  // position takes more positions a step: 500,000, k = 12: 186 / 176 / 169 / 169.
  // A cloud that the block can finish saves the other launch, so there a level may
  // have 16 Ki entries and take kWholeSteps steps of the block: 10007 points,
  // k = 1: 28.2 -> 24.0 (largest level 2346), k = 4: 34.1 -> 26.9, k = 48: 138 ->
  // 129; with eight steps it loses (30011, k = 8: 54.8 -> 66.4).
  constexpr int64_t kSmall = 1024, kSmallEntries = LANES == 1 ? 12288 : 8192;
  constexpr int64_t kWholeSteps = 5;
  const std::vector<int64_t>& lo = g->level_off_h;
  auto head_run = [&](int64_t most) {
    int a = 1;
    while (a < L && a < kHeadLevels && lo[a + 1] - lo[a] <= most && lo[a + 1] <= kHeadPoints) a++;
    return a;
  };
  int a = head_run(std::min<int64_t>(16384 / KP, kWholeSteps * (head_threads(HP) / LANES)));
  if (a < L) a = head_run(std::min(kSmall, kSmallEntries / KP));
  const int64_t* lod = g->level_off_d;
  int64_t n0 = g->n0;
  if (a > 1) {
    const size_t smem = (size_t)lo[a] * sizeof(float) + (a + 1) * sizeof(int32_t);
    auto kern = generate_head_kernel<KP, LANES>;
    GGP_CUDA(allow_dyn_smem(kern, smem));
    kern<<<1, head_threads(HP), smem, s>>>(g->nbr, f->b, f->sigma, xi, v, lod, a, n0);
    GGP_CUDA(cudaGetLastError());
  }
  if (a == L) return GRAPHGP_OK;
  // Without a barrier up to kFlowEntries row entries (barrier / flags, us): 30011
  // points, k = 16: 125 / 104; 127001, k = 7: 99 / 76; 10^6, k = 8: 168 / 143;
  // 500000, k = 16: 252 / 212; 262000, k = 32: 469 / 356; 130000, k = 64: 1058 /
  // 851.  Above, the values are no longer read soon after they are written: 10^6,
  // k = 16: 286 / 294, k = 32: 603 / 1217; 2^24, k = 16: 902 / 1098.  And only with at
  // most kFlowLevel entries a level on average, as what it saves is a barrier per
  // level: 2 x 10^6, k = 1 (24 levels): 67 / 80, k = 4 (53 levels): 124 / 91.
  const bool flow = g->N * KP <= std::min(kFlowEntries, kFlowLevel * L) && L <= kFlowMaxLevels;
  if (flow) return launch_generate_flow<KP>(g, f, xi, v, a, s);
  // the levels in between to the cooperative grid, the run of small ones at the
  // end (levels [z, L)) to one block
  constexpr int64_t kTail = 2 * small_steps(HP) * (small_threads(HP) / LANES);
  int z = L;
  while (z > a && lo[z] - lo[z - 1] <= kTail) z--;
  if (a < z) {
    GGP_CUDA(cudaMemsetAsync(g->level_bar, 0, L * sizeof(uint32_t), s));
    auto kern = generate_kernel<KP, LANES, U>;
    static int max_grid_dev[kMaxDevices] = {};
    const int max_grid = coop_grid_cached(max_grid_dev, kern, kSweepThreads);
    int64_t want = (g->max_level_size + kSweepThreads - 1) / kSweepThreads;
    int grid = (int)std::min<int64_t>(max_grid, std::max<int64_t>(want, 1));
    LevelBarrier lb{g->level_bar, g->err, g->max_spin};
    const int32_t* nbr = g->nbr;
    const float* bw = f->b;
    const float* sg = f->sigma;
    void* args[] = {(void*)&nbr, (void*)&bw, (void*)&sg, (void*)&xi, (void*)&v,
                    (void*)&lod, (void*)&a,  (void*)&z,  (void*)&n0, (void*)&lb};
    GGP_CUDA(cudaLaunchCooperativeKernel((const void*)kern, dim3(grid), dim3(kSweepThreads), args,
                                         0, s));
  }
  if (z < L) {
    generate_small_kernel<KP, LANES><<<1, small_threads(HP), 0, s>>>(g->nbr, f->b, f->sigma, xi, v,
                                                                     lod, z, L, n0);
    GGP_CUDA(cudaGetLastError());
  }
  return GRAPHGP_OK;
}

template <int KP>
int launch_whiten(graphgp_graph_t g, graphgp_factor_t f, const float* v, float* xi, double* sq,
                  cudaStream_t s) {
  int64_t n = g->N - g->n0;
  if (n <= 0) return GRAPHGP_OK;
  // A tile is one block's work, so fewer than four per SM leave the chip idle or
  // its last wave nearly empty (tiles / in order, us; k = 16): 4096 points 74 / 16,
  // 10^6 136 / 60, 2^21 (3.4 tiles per SM) 143 / 104; 2^22 (6.7 per SM) 166 / 188,
  // k = 8 92 / 98; 2^24 601 / 726: there the tile's gathers from L1 win.  k = 32: 2 x
  // 10^6 182 / 148; k = 64: 1.5 x 10^6 314 / 315.  Rows of 20 or 28 entries on one lane
  // are read in order at half the rate (U = 1, 16 bytes a lane apart), so they go to
  // tiles earlier: k = 20: 750,000 (1.2 per SM) 70 / 64, 10^6 74 / 80; k = 28: 250,000
  // (0.4 per SM) 58 / 46, 500,000 72 / 77, 10^6 103 / 134.
  constexpr int64_t kQuarterTiles = gen_lanes(KP) > 1 || KP < 20 ? 16 : (KP < 28 ? 6 : 3);
  const bool tiled = 4 * g->n_tiles >= kQuarterTiles * num_sms();
  if (tiled && g->tile_start && g->num_levels <= 8192) {
    size_t smem = (2 * (size_t)g->num_levels + 1) * sizeof(int32_t);
    GGP_CUDA(allow_dyn_smem(whiten_tiles_kernel<KP>, smem));
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, whiten_tiles_kernel<KP>, 256, smem);
    int64_t grid = std::min<int64_t>(g->n_tiles, (int64_t)std::max(per_sm, 1) * num_sms());
    whiten_tiles_kernel<KP><<<(unsigned)grid, 256, smem, s>>>(
        g->nbr, f->b, f->sigma, v, xi, g->n0, g->tile_start, g->n_tiles, g->num_levels, sq);
  } else {
    constexpr int LANES = gen_lanes(KP), U = KP / LANES <= 4 ? 2 : 1;
    const int64_t per = 256 / LANES * U;
    const int64_t grid = std::min<int64_t>((n + per - 1) / per, (int64_t)num_sms() * 8);
    whiten_flat_kernel<KP, LANES, U><<<(unsigned)grid, 256, 0, s>>>(g->nbr, f->b, f->sigma, v, xi,
                                                                    g->N, g->n0, sq);
  }
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

#define GGP_KP_DISPATCH(kp, call)            \
  switch (kp) {                              \
    case 4: call(4); break;                  \
    case 8: call(8); break;                  \
    case 12: call(12); break;                \
    case 16: call(16); break;                \
    case 20: call(20); break;                \
    case 24: call(24); break;                \
    case 28: call(28); break;                \
    case 32: call(32); break;                \
    case 48: call(48); break;                \
    default: call(64); break;                \
  }

}  // namespace

// The wait of the barrier-free sweep runs out: a point whose neighbour holds the
// not-yet mark for good.
int flow_wait_selftest(int64_t limit, uint32_t* err, cudaStream_t s) {
  Scratch sc(s);
  float* f = nullptr;    // v[2], then zeros: xi[2], sigma[2], and the weights at 8
  int32_t* nbr = nullptr;
  int64_t* off = nullptr;
  GGP_TRY(sc.alloc(&f, 12));
  GGP_TRY(sc.alloc(&nbr, 4));
  GGP_TRY(sc.alloc(&off, 3));
  const int64_t level_off[3] = {0, 1, 2};
  GGP_CUDA(cudaMemsetAsync(f, 0, 12 * sizeof(float), s));
  GGP_CUDA(cudaMemsetAsync(f, 0xff, 2 * sizeof(float), s));
  GGP_CUDA(cudaMemsetAsync(nbr, 0, 4 * sizeof(int32_t), s));
  GGP_CUDA(cudaMemcpyAsync(off, level_off, sizeof(level_off), cudaMemcpyHostToDevice, s));
  const float *b = f + 8, *sigma = f + 4, *xi = f + 2;
  int first = 1, levels = 2;
  int64_t n0 = 1;
  void* args[] = {(void*)&nbr, (void*)&b,     (void*)&sigma,  (void*)&xi, (void*)&f,    (void*)&off,
                  (void*)&first, (void*)&levels, (void*)&n0, (void*)&limit, (void*)&err};
  GGP_CUDA(cudaLaunchCooperativeKernel((const void*)generate_flow_kernel<4, 1, 2>, dim3(1),
                                       dim3(kSweepThreads), args,
                                       (2 * levels + 1) * sizeof(int32_t), s));
  return GRAPHGP_OK;
}

int dense_matvec(const float* M, const float* x, float* y, int n0, double* sq, cudaStream_t s) {
  dense_lower_matvec_kernel<<<(n0 + 7) / 8, 256, 0, s>>>(M, x, y, n0, sq);
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

int run_generate(graphgp_graph_t g, graphgp_factor_t f, const float* xi, float* v,
                 cudaStream_t s) {
  int n0 = g->n0;
  dense_lower_matvec_kernel<<<(n0 + 7) / 8, 256, 0, s>>>(f->L0, xi, v, n0, nullptr);
  GGP_CUDA(cudaGetLastError());
  int rc = GRAPHGP_OK;
#define GGP_GEN(KP) rc = launch_generate<KP>(g, f, xi, v, s)
  GGP_KP_DISPATCH(g->kp, GGP_GEN)
#undef GGP_GEN
  return rc;
}

int run_whiten(graphgp_graph_t g, graphgp_factor_t f, const float* v, float* xi, double* sq,
               cudaStream_t s) {
  int n0 = g->n0;
  dense_lower_matvec_kernel<<<(n0 + 7) / 8, 256, 0, s>>>(f->L0inv, v, xi, n0, sq);
  GGP_CUDA(cudaGetLastError());
  int rc = GRAPHGP_OK;
#define GGP_WH(KP) rc = launch_whiten<KP>(g, f, v, xi, sq, s)
  GGP_KP_DISPATCH(g->kp, GGP_WH)
#undef GGP_WH
  return rc;
}

}  // namespace ggp

using namespace ggp;

static bool same_graph(graphgp_graph_t g, graphgp_factor_t f) {
  return g && f && f->g == g && f->row_end < 0;  // whole-graph factors only
}

extern "C" int graphgp_generate(graphgp_graph_t g, graphgp_factor_t f, const float* xi_d,
                                float* v_d, void* stream) {
  if (!same_graph(g, f) || !xi_d || !v_d) return GRAPHGP_ERR_INVALID;
  if (xi_d < v_d + g->N && v_d < xi_d + g->N) return GRAPHGP_ERR_INVALID;  // overlap
  return run_generate(g, f, xi_d, v_d, (cudaStream_t)stream);
}

extern "C" int graphgp_whiten(graphgp_graph_t g, graphgp_factor_t f, const float* v_d,
                              float* xi_d, void* stream) {
  if (!same_graph(g, f) || !xi_d || !v_d) return GRAPHGP_ERR_INVALID;
  return run_whiten(g, f, v_d, xi_d, nullptr, (cudaStream_t)stream);
}

extern "C" int graphgp_logdet(graphgp_factor_t f, double* out_d, void* stream) {
  if (!f || !out_d) return GRAPHGP_ERR_INVALID;
  GGP_CUDA(cudaMemcpyAsync(out_d, f->logdet, sizeof(double), cudaMemcpyDeviceToDevice,
                           (cudaStream_t)stream));
  return GRAPHGP_OK;
}

extern "C" int graphgp_nll(graphgp_graph_t g, graphgp_factor_t f, const float* v_d,
                           double* out_d, void* stream) {
  if (!same_graph(g, f) || !v_d || !out_d) return GRAPHGP_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  Scratch sc(s);
  double* sq = nullptr;
  GGP_TRY(sc.alloc(&sq, 1));
  GGP_CUDA(cudaMemsetAsync(sq, 0, 8, s));
  GGP_TRY(run_whiten(g, f, v_d, g->tmp_vec, sq, s));
  nll_finish_kernel<<<1, 1, 0, s>>>(sq, f->logdet, out_d);
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

extern "C" int graphgp_sync_status(graphgp_graph_t g, graphgp_factor_t f, void* stream,
                                   int64_t* n_not_pd) {
  GGP_CUDA(cudaStreamSynchronize((cudaStream_t)stream));
  uint32_t err = 0;
  unsigned long long bad = 0;
  if (g) GGP_CUDA(cudaMemcpy(&err, g->err, 4, cudaMemcpyDeviceToHost));
  if (f) GGP_CUDA(cudaMemcpy(&bad, f->not_pd, 8, cudaMemcpyDeviceToHost));
  if (n_not_pd) *n_not_pd = (int64_t)bad;
  if (err & ERRBIT_TIMEOUT) return GRAPHGP_ERR_TIMEOUT;
  if (err & ERRBIT_INDEX) return GRAPHGP_ERR_INVALID;
  if (bad) return GRAPHGP_WARN_NOT_PD;
  return GRAPHGP_OK;
}

extern "C" const char* graphgp_status_string(int status) {
  switch (status) {
    case GRAPHGP_OK: return "ok";
    case GRAPHGP_ERR_INVALID: return "invalid argument";
    case GRAPHGP_ERR_OOM: return "device out of memory";
    case GRAPHGP_ERR_CUDA: return "CUDA runtime error";
    case GRAPHGP_ERR_TIMEOUT: return "bounded device wait timed out";
    case GRAPHGP_ERR_NAN: return "non-finite input";
    case GRAPHGP_ERR_IO: return "file error";
    case GRAPHGP_WARN_NOT_PD: return "pivots clamped (matrix not positive definite)";
  }
  return "unknown status";
}
