// Preceding k-nearest-neighbour search (Sec. 2.1: c(i) = the k nearest
// preceding points; Sec. 2.2: every prefix of the tree order is itself a
// valid tree, so the points preceding tree index j are searched in the
// prefix tree {0..j-1}).
//
// One warp searches for 32 spatially adjacent queries of one tree level
// together: it walks the tree once, with one stack, and visits a node when the
// node's bounding box is near enough for any of them.  Control flow and node
// loads are uniform, every visited point is tested by all lanes, and points
// that pass a lane's current k-th key go to a short queue of that lane in
// shared memory; when a queue is full all lanes merge theirs into their sorted
// lists (a bitonic sort and merge for k <= 16).  One query per thread spent its
// time in divergence: whenever any lane inserted, the warp ran the whole
// insertion, and each lane fetched other nodes.  Bound by instruction issue
// (about 70,000 per warp of queries).  2^22 clustered points, k = 16: 21.4 ms
// with one query per thread and splitting planes, 13.5 ms here; testing the
// lowest three tree levels without boxes and deferring a node's own point until
// its nearer child is done gave 2 ms of it, a queue of a whole list little.
//
// Nodes are stored in heap order: node h on level l (2^l <= h < 2^(l+1)) has
// children 2 h and 2 h + 1, so siblings share a memory sector; its tree index
// is 2^l - 1 + bitrev_l(h - 2^l), the bit-reversed layout of Sec. 2.2.  A
// level's queries in heap order are in k-d in-order, hence adjacent.
//
// A box is skipped for a lane only if the FP32 key of its nearest corner,
// formed with the operations of the point key d2 = fma(dz,dz, fma(dy,dy,
// dx*dx)) from offsets no larger than those of any point in the box, exceeds
// the lane's k-th key; IEEE rounding is monotone, so no point inside can have
// a smaller key and the result is exactly the brute-force definition: the k
// smallest (d2, tree index).
#include <algorithm>

#include "common.cuh"

namespace ggp {
namespace {

// bitrev_l(h - 2^l): the position on its level of heap node h, h < 2^32 as
// N < 2^31 (reversing h puts its leading bit right below the others).
__device__ __forceinline__ uint32_t level_position(uint32_t h, int l) {
  return __brev(h) >> (31 - l) >> 1;
}

__global__ void heap_points_kernel(const float* __restrict__ pts,
                                   const int32_t* __restrict__ tree_point, int64_t N,
                                   float4* __restrict__ hx) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < N;
       j += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = tree_point[j];
    hx[tree_heap_index(j)] = make_float4(pts[3 * p], pts[3 * p + 1], pts[3 * p + 2], 0.0f);
  }
}

__device__ __forceinline__ float key_d2(float dx, float dy, float dz) {
  return __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
}

// Largest offset-wise lower bound of the key of any point in the box.
__device__ __forceinline__ float box_key(float4 lo, float4 hi, float4 q) {
  const float dx = fmaxf(fmaxf(__fsub_rn(lo.x, q.x), __fsub_rn(q.x, hi.x)), 0.0f);
  const float dy = fmaxf(fmaxf(__fsub_rn(lo.y, q.y), __fsub_rn(q.y, hi.y)), 0.0f);
  const float dz = fmaxf(fmaxf(__fsub_rn(lo.z, q.z), __fsub_rn(q.z, hi.z)), 0.0f);
  return key_d2(dx, dy, dz);
}

// Sorted list of KM (key, index) entries as 64-bit integers (keys are
// non-negative floats, whose bits order as integers).  The first KM - k
// entries are zero fillers, which no real entry precedes, so the k real
// entries always sit in the last k slots and the k-th is entry KM - 1.
// Queued candidates per lane: a whole list for KM <= 16.
__host__ __device__ constexpr int queue_len(int km) { return km <= 16 ? km : 16; }

__device__ __forceinline__ void exchange(unsigned long long& a, unsigned long long& b, bool up) {
  const bool sw = (b < a) == up;
  const unsigned long long t = sw ? a : b;
  a = sw ? b : a;
  b = t;
}

// Bitonic stages on Q entries: from span `size` to 2 (ascending).
template <int Q>
__device__ __forceinline__ void bitonic_merge(unsigned long long (&e)[Q]) {
#pragma unroll
  for (int d = Q / 2; d; d /= 2)
#pragma unroll
    for (int i = 0; i < Q; i++)
      if (!(i & d)) exchange(e[i], e[i | d], true);
}

template <int Q>
__device__ __forceinline__ void bitonic_sort(unsigned long long (&e)[Q]) {
#pragma unroll
  for (int size = 2; size <= Q; size *= 2)
#pragma unroll
    for (int d = size / 2; d; d /= 2)
#pragma unroll
      for (int i = 0; i < Q; i++)
        if (!(i & d)) exchange(e[i], e[i | d], size == Q || !(i & size));
}

template <int KM>
__device__ __forceinline__ void list_insert(unsigned long long (&e)[KM], unsigned long long c) {
#pragma unroll
  for (int m = KM - 1; m > 0; m--)
    e[m] = c < e[m - 1] ? e[m - 1] : (c < e[m] ? c : e[m]);
  e[0] = c < e[0] ? c : e[0];
}

template <int KM>
__global__ void __launch_bounds__(128) knn_kernel(
    const float4* __restrict__ hx, const float4* __restrict__ box, int64_t N, int k, int64_t n0,
    int levels, int64_t t_first, int64_t t_end, int last_shift, int32_t* __restrict__ nbr_tree,
    uint32_t* __restrict__ err) {
  constexpr int Q = queue_len(KM);
  __shared__ unsigned long long queue[Q][128];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int64_t t = t_first + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  // slot t is heap node t, except on a sparse last level, whose existing nodes
  // are every 2^last_shift-th
  uint32_t j = 0;  // tree index of the lane's query (never 0 for one that exists)
  float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
  if (t < t_end) {
    uint32_t h = (uint32_t)t;
    const int l = 31 - __clz(h);
    if (l == levels - 1) h = (1u << l) + ((h - (1u << l)) << last_shift);
    j = (1u << l) - 1 + level_position(h, l);
    if (j >= (uint32_t)N || j < (uint32_t)n0) j = 0;
    if (j) q = hx[h];
  }
  const uint32_t jmax = __reduce_max_sync(full, j);
  if (!jmax) return;  // no query in this warp
  // Lanes without a query vote on the order of the walk, so they take the place of
  // the nearest query below (else the first) and vote with it.  On a half-empty last
  // level, left at the origin they sent every warp to that end of the cloud first:
  // along a line each point on the way back then enters the lists (200,000 points, d
  // = 1, k = 8: 56 ms for the build, 1.8 without them).
  {
    const unsigned has = __ballot_sync(full, j != 0), below = has & ((2u << lane) - 1u);
    const int src = below ? 31 - __clz(below) : __ffs(has) - 1;
    q.x = __shfl_sync(full, q.x, src);
    q.y = __shfl_sync(full, q.y, src);
    q.z = __shfl_sync(full, q.z, src);
  }
  unsigned long long e[KM];
#pragma unroll
  for (int a = 0; a < KM; a++) e[a] = a < KM - k ? 0ull : 0x7f8000007fffffffull;
  float kth = j ? __int_as_float(0x7f800000) : -1.0f;  // key of the k-th entry
  unsigned kid = 0x7fffffffu;                                 // its index
  int cnt = 0;
  auto flush = [&]() {
    if constexpr (KM <= 16) {  // sort the queue, keep the KM smallest of both
      unsigned long long c[Q];
#pragma unroll
      for (int i = 0; i < Q; i++) c[i] = i < cnt ? queue[i][threadIdx.x] : ~0ull;
      bitonic_sort<Q>(c);
#pragma unroll
      for (int i = 0; i < KM; i++) e[i] = c[Q - 1 - i] < e[i] ? c[Q - 1 - i] : e[i];
      bitonic_merge<KM>(e);
    } else {
      int most = cnt;
      for (int o = 16; o; o >>= 1) most = max(most, __shfl_xor_sync(full, most, o));
      for (int i = 0; i < most; i++) {
        const unsigned long long c = i < cnt ? queue[i][threadIdx.x] : ~0ull;
        if (__any_sync(full, c < e[KM - 1])) list_insert<KM>(e, c);
      }
    }
    cnt = 0;
    if (j) {
      kth = __int_as_float((int)(e[KM - 1] >> 32));
      kid = (unsigned)e[KM - 1];
    }
  };
  auto test_point = [&](float4 x, uint32_t idx) {  // candidate idx at x
    const float d = key_d2(__fsub_rn(x.x, q.x), __fsub_rn(x.y, q.y), __fsub_rn(x.z, q.z));
    if (idx < j && (d < kth || (d == kth && idx < kid))) {
      queue[cnt][threadIdx.x] = ((unsigned long long)__float_as_uint(d) << 32) | idx;
      cnt++;
    }
    if (__any_sync(full, cnt == Q)) flush();
  };
  // Depth-first, the nearer child first; a node's own point is tested after
  // its nearer child (on the way down it would enter every list only to be
  // replaced).  Pending work is keyed by the node's level, at most one point
  // and one farther child each, and held one level per lane.
  uint32_t points = 0, children = 0;    // lane l: node / child pending at level l
  uint32_t has_point = 0, has_child = 0;  // the same as masks over levels (uniform)
  uint32_t h = 1;  // the root; always visited
  int l = 0;
  while (true) {
    const uint32_t pos = level_position(h, l);
    const uint32_t i0 = (2u << l) - 1 + pos, i1 = i0 + (1u << l), c0 = 2 * h;  // the children
    uint32_t next = 0;
    if (l + 2 >= levels - 1) {
      // the lowest three levels: testing the (at most seven) points costs less
      // than the boxes that would spare some of them
      test_point(__ldg(hx + h), i0 - (1u << l));
      if (l + 1 < levels) {
        if (i0 < jmax) test_point(__ldg(hx + c0), i0);
        if (i1 < jmax) test_point(__ldg(hx + c0 + 1), i1);
        if (l + 2 < levels) {
          const uint32_t g0 = (4u << l) - 1 + pos, w = 1u << l;  // grandchildren 4 h + (0, 2, 1, 3)
          if (g0 < jmax) test_point(__ldg(hx + 2 * c0), g0);
          if (g0 + w < jmax) test_point(__ldg(hx + 2 * c0 + 2), g0 + w);
          if (g0 + 2 * w < jmax) test_point(__ldg(hx + 2 * c0 + 1), g0 + 2 * w);
          if (g0 + 3 * w < jmax) test_point(__ldg(hx + 2 * c0 + 3), g0 + 3 * w);
        }
      }
    } else {
      const float4* b = box + 2 * (size_t)c0;
      const float b0 = box_key(__ldg(b), __ldg(b + 1), q), b1 = box_key(__ldg(b + 2), __ldg(b + 3), q);
      const bool near0 = __any_sync(full, i0 < j && b0 <= kth);
      const bool near1 = __any_sync(full, i1 < j && b1 <= kth);
      if (near0 && near1) {
        const bool left = 2 * __popc(__ballot_sync(full, b0 <= b1)) >= 32;
        next = left ? c0 : c0 + 1;
        if (lane == l) children = left ? c0 + 1 : c0;
        has_child |= 1u << l;
      } else if (near0 || near1) {
        next = near0 ? c0 : c0 + 1;
      }
      if (lane == l) points = h;
      has_point |= 1u << l;
      l++;
    }
    while (!next && (has_point | has_child)) {  // the deepest pending work
      const int lv = 31 - __clz(has_point | has_child);
      if ((has_point >> lv) & 1) {
        has_point &= ~(1u << lv);
        const uint32_t p = __shfl_sync(full, points, lv);
        test_point(__ldg(hx + p), (1u << lv) - 1 + level_position(p, lv));
      } else {
        has_child &= ~(1u << lv);
        const uint32_t c = __shfl_sync(full, children, lv);
        const float b = box_key(__ldg(box + 2 * (size_t)c), __ldg(box + 2 * (size_t)c + 1), q);
        if (__any_sync(full, b <= kth)) {
          next = c;
          l = lv + 1;
        }
      }
    }
    if (!next) break;
    h = next;
  }
  flush();
  if (!j) return;
  int32_t* out = nbr_tree + ((int64_t)j - n0) * k;
#pragma unroll
  for (int a = 0; a < KM; a++)
    if (a >= KM - k) {
      int32_t id = (int32_t)(uint32_t)e[a];
      if (id < 0 || (uint32_t)id >= j) {  // cannot happen for n0 >= k; guards later gathers
        id = 0;
        atomicOr(err, ERRBIT_INDEX);
      }
      out[a - (KM - k)] = id;
    }
}

}  // namespace

int knn_query(const float* pts, const int32_t* tree_point, const float4* box, int64_t N, int k,
              int64_t n0, int32_t* nbr_tree, uint32_t* err, cudaStream_t s) {
  if (N <= n0) return GRAPHGP_OK;
  int levels = 0;
  while (((int64_t(1) << levels) - 1) < N) levels++;
  Scratch sc(s);
  float4* hx = nullptr;
  GGP_TRY(sc.alloc(&hx, (size_t)1 << levels));
  heap_points_kernel<<<grid_for(N, 256), 256, 0, s>>>(pts, tree_point, N, hx);
  GGP_CUDA(cudaGetLastError());
  // slots: the heap nodes from the level of n0 on; of the last level only the
  // multiples of 2^last_shift that can exist (tree positions below its count).  At
  // most kMaxShift, so that a warp's queries stay within 1024 neighbouring nodes: of
  // queries far apart some are searched for from the wrong end (131,073 points along
  // a line, two on the last level: 22.6 ms, one warp's walk over the whole tree).
  int l0 = 0;
  while (((int64_t(2) << l0) - 1) <= n0) l0++;
  const int last = levels - 1;
  const int64_t count = N - ((int64_t(1) << last) - 1);
  int bits = 0;
  while ((int64_t(1) << bits) < count) bits++;
  constexpr int kMaxShift = 5;
  const int last_shift = std::min(last - bits, kMaxShift);
  const int64_t t_first = int64_t(1) << l0;
  const int64_t t_end = (int64_t(1) << last) + (int64_t(1) << (last - last_shift));
  const int B = 128;
  const unsigned grid = (unsigned)((t_end - t_first + B - 1) / B);
#define GGP_KNN(KM)                                                                            \
  knn_kernel<KM><<<grid, B, 0, s>>>(hx, box, N, k, n0, levels, t_first, t_end, last_shift,     \
                                    nbr_tree, err)
  if (k <= 8) GGP_KNN(8);
  else if (k <= 16) GGP_KNN(16);
  else if (k <= 32) GGP_KNN(32);
  else GGP_KNN(64);
#undef GGP_KNN
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

}  // namespace ggp
