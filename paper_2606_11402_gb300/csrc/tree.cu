// Left-balanced k-d tree in the bit-reversed layout (Sec. 2.2 "Tree
// ordering", "Bit-reversed ordering"; Sec. 2.3: sort-based GPU build).
//
// Design: the points are sorted once per dimension by (coordinate, input
// index).  The three sorted orders are kept, each restricted to every open
// subtree, in the subtree's in-order slot range.  Processing the tree one
// level at a time:
//   * the bounding box of a subtree is read off the ends of its three sorted
//     ranges (no reduction), which fixes the split dimension;
//   * the median of the split dimension is the element at offset m (the size
//     of the left subtree) of that dimension's range: no selection pass;
//   * the two other orders are stably partitioned (left part, node, right
//     part) with one exclusive scan each, so they stay sorted.
// Once a subtree has at most kSub nodes, one block takes it through all of its
// levels in shared memory (tree_sub_kernel).
// Every step is a permutation fixed by the data, so the result is exactly
// the recursive definition: split on the widest FP32 extent (ties to the
// lowest dimension) or on level mod 3, median by (coordinate, input index).
#include "common.cuh"

namespace ggp {
namespace {

__device__ __forceinline__ int node_level(int64_t j) {
  return 63 - __clzll((unsigned long long)(j + 1));
}

// Number of existing nodes in the subtree at (level l, position p): the
// descendants on level m occupy positions p + t 2^l, t < 2^(m-l); every level but
// the last is full.
__host__ __device__ __forceinline__ int64_t subtree_nodes(int64_t p, int l, int64_t N, int levels) {
  if (l >= levels) return 0;
  const int64_t cap = int64_t(1) << (levels - 1 - l);
  const int64_t rest = N - ((int64_t(1) << (levels - 1)) - 1 + p);
  if (rest <= 0) return cap - 1;
  const int64_t n = ((rest - 1) >> l) + 1;
  return cap - 1 + (n < cap ? n : cap);
}

__device__ __forceinline__ uint32_t orderable(float f) {
  uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__global__ void presort_keys_kernel(const float* __restrict__ pts, int64_t N,
                                    int dim, uint32_t* __restrict__ keys,
                                    uint32_t* __restrict__ ids) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N;
       i += (int64_t)gridDim.x * blockDim.x) {
    keys[i] = orderable(pts[3 * i + dim]);
    ids[i] = (uint32_t)i;
  }
}

struct Orders {
  const int32_t* o[3];
};

// One thread per node of level l: split dimension, median point, in-order
// rank, and the in-order start of both children.
__global__ void level_nodes_kernel(const float* __restrict__ pts, int64_t N,
                                   int l, int levels, int rule, Orders ord,
                                   int32_t* __restrict__ start,
                                   int32_t* __restrict__ msize,
                                   int32_t* __restrict__ tree_point,
                                   uint8_t* __restrict__ split_dim,
                                   int32_t* __restrict__ inorder,
                                   int32_t* __restrict__ node_at_inorder,
                                   float4* __restrict__ box) {
  int64_t first = (int64_t(1) << l) - 1;
  int64_t count = int64_t(1) << l;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < count;
       t += (int64_t)gridDim.x * blockDim.x) {
    int64_t j = first + t;
    if (j >= N) return;
    int64_t S = subtree_nodes(t, l, N, levels);
    int64_t lc = j + (int64_t(1) << l), rc = j + (int64_t(2) << l);
    int64_t m = subtree_nodes(t, l + 1, N, levels);
    int64_t st = start[j];
    int dim;
    float lo[3], hi[3], ext[3];
    if (rule == 0 || box) {
#pragma unroll
      for (int d = 0; d < 3; d++) {
        lo[d] = pts[3 * (int64_t)ord.o[d][st] + d];
        hi[d] = pts[3 * (int64_t)ord.o[d][st + S - 1] + d];
        ext[d] = __fsub_rn(hi[d], lo[d]);
      }
    }
    if (box) {
      const int64_t h = tree_heap_index(j);
      box[2 * h] = make_float4(lo[0], lo[1], lo[2], 0.0f);
      box[2 * h + 1] = make_float4(hi[0], hi[1], hi[2], 0.0f);
    }
    if (rule == 0) {
      dim = 0;
      if (ext[1] > ext[dim]) dim = 1;
      if (ext[2] > ext[dim]) dim = 2;
    } else {
      dim = l % 3;
    }
    int32_t p = ord.o[dim][st + m];
    tree_point[j] = p;
    split_dim[j] = (uint8_t)dim;
    inorder[j] = (int32_t)(st + m);
    msize[j] = (int32_t)m;
    node_at_inorder[st + m] = (int32_t)j;
    if (lc < N) start[lc] = (int32_t)st;
    if (rc < N) start[rc] = (int32_t)(st + m + 1);
  }
}

// One thread per in-order slot: the side (0 left, 1 node, 2 right) of the
// element found in the split dimension's order, and the slot's subtree on
// the next level (-1 once it holds a finished node).
__global__ void slot_side_kernel(int64_t N, Orders ord,
                                 const int32_t* __restrict__ seg,
                                 int32_t* __restrict__ seg_next,
                                 const int32_t* __restrict__ start,
                                 const int32_t* __restrict__ msize,
                                 const uint8_t* __restrict__ split_dim,
                                 uint8_t* __restrict__ side) {
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < N;
       x += (int64_t)gridDim.x * blockDim.x) {
    int32_t j = seg[x];
    if (j < 0) {
      seg_next[x] = -1;
      continue;
    }
    int64_t r = x - start[j];
    int64_t m = msize[j];
    int l = node_level(j);
    int32_t e = ord.o[split_dim[j]][x];
    uint8_t sd = r < m ? 0 : (r == m ? 1 : 2);
    side[e] = sd;
    seg_next[x] = sd == 0 ? (int32_t)(j + (int64_t(1) << l))
                          : (sd == 1 ? -1 : (int32_t)(j + (int64_t(2) << l)));
  }
}

// Flags of the elements that go left in the order of dimension A = A0 +
// blockIdx.y, inside subtrees that do not split on A; records the slot of each
// node element.  flags and node_slot hold N entries per dimension of the launch.
__global__ void part_flags_kernel(int64_t N, int A0, Orders ord, const int32_t* __restrict__ seg,
                                  const uint8_t* __restrict__ split_dim,
                                  const uint8_t* __restrict__ side,
                                  uint32_t* __restrict__ flags,
                                  int32_t* __restrict__ node_slot) {
  const int A = A0 + blockIdx.y;
  const int32_t* ordA = ord.o[A];
  flags += blockIdx.y * N;
  node_slot += blockIdx.y * N;
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < N;
       x += (int64_t)gridDim.x * blockDim.x) {
    int32_t j = seg[x];
    uint32_t f = 0;
    if (j >= 0 && split_dim[j] != A) {
      uint8_t sd = side[ordA[x]];
      f = sd == 0;
      if (sd == 1) node_slot[j] = (int32_t)x;
    }
    flags[x] = f;
  }
}

struct OrdersOut {
  int32_t* o[3];
};

// pre: exclusive prefix of flags over all dimensions of the launch; only
// differences within one dimension are used.
__global__ void part_scatter_kernel(int64_t N, int A0, Orders ord, OrdersOut next,
                                    const int32_t* __restrict__ seg,
                                    const uint8_t* __restrict__ split_dim,
                                    const uint8_t* __restrict__ side,
                                    const uint32_t* __restrict__ pre,
                                    const int32_t* __restrict__ start,
                                    const int32_t* __restrict__ msize,
                                    const int32_t* __restrict__ node_slot) {
  const int A = A0 + blockIdx.y;
  const int32_t* ordA = ord.o[A];
  int32_t* ordA_next = next.o[A];
  pre += blockIdx.y * N;
  node_slot += blockIdx.y * N;
  for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < N;
       x += (int64_t)gridDim.x * blockDim.x) {
    int32_t j = seg[x];
    int32_t e = ordA[x];
    int64_t dest = x;
    if (j >= 0 && split_dim[j] != A) {
      int64_t st = start[j];
      int64_t m = msize[j];
      int64_t lr = (int64_t)(pre[x] - pre[st]);
      uint8_t sd = side[e];
      if (sd == 0) {
        dest = st + lr;
      } else if (sd == 1) {
        dest = st + m;
      } else {
        int64_t nb = node_slot[j] < x ? 1 : 0;
        dest = st + m + 1 + ((x - st) - lr - nb);
      }
    }
    ordA_next[dest] = e;
  }
}

// ---- subtrees of at most kSub nodes -------------------------------------------
// One block per subtree of level l0, one thread per slot: the three orders, as
// 16-bit indices into the block's points, stay in shared memory for the
// remaining levels, which would each cost a device-wide pass over six arrays
// (about 1.1 ms at 2^24 points, and seventeen launches at any size).  The same
// medians and stable partitions as above, so the same tree.  Bound by the block
// barriers, six a level.  The ten levels of 2^24 points take 2.3 ms, 11 ms by
// passes; a whole build of 30011 points goes from 2.37 to 1.44 ms.
constexpr int kSub = 1024;

struct SubTree {
  float x[3][kSub];
  int32_t gid[kSub];
  uint16_t ord[2][3][kSub];        // [level parity][dimension][slot]
  uint16_t seg[2][kSub];           // node of the slot on this level, kNone once done
  uint16_t start[2][kSub], size[2][kSub];
  uint16_t m[kSub], pre[3][kSub], slot[3][kSub];
  uint16_t wsum[3][kSub / 32];
  uint8_t dim[kSub], side[kSub];
};
constexpr uint16_t kNone = 0xffff;

__global__ void __launch_bounds__(kSub, 2) tree_sub_kernel(
    const float* __restrict__ pts, int64_t N, int l0, int levels, int rule, Orders ord,
    const int32_t* __restrict__ start, int32_t* loc, int32_t* __restrict__ tree_point,
    uint8_t* __restrict__ split_dim, int32_t* __restrict__ inorder,
    int32_t* __restrict__ node_at_inorder, float4* __restrict__ box) {
  extern __shared__ __align__(16) unsigned char sub_smem[];
  SubTree& T = *reinterpret_cast<SubTree*>(sub_smem);
  const int x = threadIdx.x, lane = x & 31, warp = x >> 5;
  const int64_t p = blockIdx.x, j0 = (int64_t(1) << l0) - 1 + p;
  if (j0 >= N) return;
  const int S0 = (int)subtree_nodes(p, l0, N, levels);
  const int64_t st0 = start[j0];
  if (x < S0) {
    const int32_t e = ord.o[0][st0 + x];
    T.gid[x] = e;
    for (int d = 0; d < 3; d++) T.x[d][x] = pts[3 * (int64_t)e + d];
    T.ord[0][0][x] = (uint16_t)x;
    loc[e] = x;
  }
  T.seg[0][x] = x < S0 ? 0 : kNone;
  if (x == 0) {
    T.start[0][0] = 0;
    T.size[0][0] = (uint16_t)S0;
  }
  __syncthreads();
  if (x < S0)
    for (int d = 1; d < 3; d++) T.ord[0][d][x] = (uint16_t)loc[ord.o[d][st0 + x]];
  __syncthreads();
  for (int l = l0; l < levels; l++) {
    const int c = (l - l0) & 1, nodes = 1 << (l - l0);
    if (x < nodes) {  // the nodes of this level
      const int64_t pos = p + ((int64_t)x << l0), j = (int64_t(1) << l) - 1 + pos;
      if (j < N) {
        const int S = T.size[c][x], st = T.start[c][x];
        const int m = (int)subtree_nodes(pos, l + 1, N, levels);
        float lo[3], hi[3], ext[3];
        for (int d = 0; d < 3; d++) {
          lo[d] = T.x[d][T.ord[c][d][st]];
          hi[d] = T.x[d][T.ord[c][d][st + S - 1]];
          ext[d] = __fsub_rn(hi[d], lo[d]);
        }
        int dim = l % 3;
        if (rule == 0) {
          dim = ext[1] > ext[0] ? 1 : 0;
          if (ext[2] > (dim ? ext[1] : ext[0])) dim = 2;
        }
        if (box && l < levels - 2) {
          const int64_t h = tree_heap_index(j);
          box[2 * h] = make_float4(lo[0], lo[1], lo[2], 0.0f);
          box[2 * h + 1] = make_float4(hi[0], hi[1], hi[2], 0.0f);
        }
        tree_point[j] = T.gid[T.ord[c][dim][st + m]];
        split_dim[j] = (uint8_t)dim;
        inorder[j] = (int32_t)(st0 + st + m);
        node_at_inorder[st0 + st + m] = (int32_t)j;
        T.m[x] = (uint16_t)m;
        T.dim[x] = (uint8_t)dim;
        if (m > 0) {
          T.start[c ^ 1][x] = (uint16_t)st;
          T.size[c ^ 1][x] = (uint16_t)m;
        }
        if (S - 1 - m > 0) {
          T.start[c ^ 1][x + nodes] = (uint16_t)(st + m + 1);
          T.size[c ^ 1][x + nodes] = (uint16_t)(S - 1 - m);
        }
      }
    }
    if (l == levels - 1) break;
    __syncthreads();
    const int t = T.seg[c][x];  // this slot's node; its split dimension's order
    int st = 0, m = 0, dim = 3;
    if (t != kNone) {
      st = T.start[c][t];
      m = T.m[t];
      dim = T.dim[t];
      const int r = x - st;
      const int sd = r < m ? 0 : (r == m ? 1 : 2);
      T.side[T.ord[c][dim][x]] = (uint8_t)sd;
      T.seg[c ^ 1][x] = sd == 1 ? kNone : (uint16_t)(sd == 0 ? t : t + nodes);
    } else {
      T.seg[c ^ 1][x] = kNone;
    }
    __syncthreads();
    int sides = 0;  // two bits per dimension
#pragma unroll
    for (int A = 0; A < 3; A++) {
      int sd = 3;
      if (t != kNone && dim != A) {
        sd = T.side[T.ord[c][A][x]];
        if (sd == 1) T.slot[A][t] = (uint16_t)x;
      }
      sides |= sd << (2 * A);
      const unsigned left = __ballot_sync(0xffffffffu, sd == 0);
      T.pre[A][x] = (uint16_t)__popc(left & ((1u << lane) - 1u));
      if (lane == 0) T.wsum[A][warp] = (uint16_t)__popc(left);
    }
    __syncthreads();
    if (warp < 3) {  // exclusive scan of the warps' counts
      const int v = T.wsum[warp][lane];
      int s = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += y;
      }
      T.wsum[warp][lane] = (uint16_t)(s - v);
    }
    __syncthreads();
    if (t != kNone) {
#pragma unroll
      for (int A = 0; A < 3; A++) {
        const uint16_t e = T.ord[c][A][x];
        int dest = x;
        if (dim != A) {
          const int lr = T.pre[A][x] + T.wsum[A][warp] - T.pre[A][st] - T.wsum[A][st >> 5];
          const int sd = (sides >> (2 * A)) & 3;
          dest = sd == 0 ? st + lr
                         : (sd == 1 ? st + m
                                    : st + m + 1 + (x - st) - lr - (T.slot[A][t] < x ? 1 : 0));
        }
        T.ord[c ^ 1][A][dest] = e;
      }
    }
    __syncthreads();
  }
}

}  // namespace

int tree_build(const float* pts, int64_t N, int rule, int32_t* tree_point,
               uint8_t* split_dim, int32_t* inorder, int32_t* node_at_inorder,
               float4* box, cudaStream_t s) {
  if (N <= 0) return GRAPHGP_OK;
  Scratch sc(s);
  // The levels down to the first whose subtrees fit a block, then those in blocks.
  int levels = 0, l0 = 0;
  while (((int64_t(1) << levels) - 1) < N) levels++;
  while (subtree_nodes(0, l0, N, levels) > kSub) l0++;
  // Up to kBatch points the three partitions of a level share their launches
  // (seven instead of seventeen a level, each a few us); above, the passes are
  // bound by memory and one dimension's scratch serves all three.
  constexpr int64_t kBatch = int64_t(1) << 21;
  const int nb = N <= kBatch ? 3 : 1;
  // Scratch, 45 bytes per point above kBatch: with the boxes (8 to 16) and
  // node_at_inorder the build's peak stays below 70.  The presort's three arrays
  // serve the partitions afterwards; start and msize hold the nodes of the levels
  // done by passes and of the first done in blocks.
  int32_t* ord[3][2];
  uint32_t *keys = nullptr, *keys_sorted = nullptr, *ids = nullptr;
  for (int d = 0; d < 3; d++)
    for (int h = 0; h < 2; h++) GGP_TRY(sc.alloc(&ord[d][h], N));
  GGP_TRY(sc.alloc(&keys, nb * N));
  GGP_TRY(sc.alloc(&keys_sorted, nb * N));
  GGP_TRY(sc.alloc(&ids, nb * N));
  const int B = 256;
  const unsigned grid = grid_for(N, B);
  for (int d = 0; d < 3; d++) {
    presort_keys_kernel<<<grid, B, 0, s>>>(pts, N, d, keys, ids);
    GGP_CUDA(cudaGetLastError());
    GGP_TRY(radix_sort_pairs(keys, ids, keys_sorted, (uint32_t*)ord[d][0], N, 32, s));
  }
  uint32_t *flags = keys, *pre = keys_sorted;
  int32_t* node_slot = (int32_t*)ids;
  int32_t *seg[2], *start = nullptr, *msize = nullptr;
  uint8_t* side = nullptr;
  GGP_TRY(sc.alloc(&seg[0], N));
  GGP_TRY(sc.alloc(&seg[1], N));
  GGP_TRY(sc.alloc(&start, (size_t)2 << l0));
  GGP_TRY(sc.alloc(&msize, (size_t)1 << l0));
  GGP_TRY(sc.alloc(&side, N));
  GGP_CUDA(cudaMemsetAsync(seg[0], 0, N * sizeof(int32_t), s));  // all in root
  GGP_CUDA(cudaMemsetAsync(start, 0, sizeof(int32_t), s));
  int cur = 0;
  for (int l = 0; l < l0; l++) {
    Orders o;
    OrdersOut next;
    for (int d = 0; d < 3; d++) {
      o.o[d] = ord[d][cur];
      next.o[d] = ord[d][1 - cur];
    }
    int64_t nodes = int64_t(1) << l;
    level_nodes_kernel<<<grid_for(nodes, B), B, 0, s>>>(pts, N, l, levels, rule, o, start, msize,
                                                        tree_point, split_dim, inorder,
                                                        node_at_inorder, box);
    GGP_CUDA(cudaGetLastError());
    slot_side_kernel<<<grid, B, 0, s>>>(N, o, seg[cur], seg[1 - cur], start, msize, split_dim,
                                        side);
    GGP_CUDA(cudaGetLastError());
    for (int A = 0; A < 3; A += nb) {
      part_flags_kernel<<<dim3(grid, nb), B, 0, s>>>(N, A, o, seg[cur], split_dim, side, flags,
                                                     node_slot);
      GGP_CUDA(cudaGetLastError());
      GGP_TRY(scan_exclusive_u32(flags, pre, nb * N, s));
      part_scatter_kernel<<<dim3(grid, nb), B, 0, s>>>(N, A, o, next, seg[cur], split_dim, side,
                                                       pre, start, msize, node_slot);
      GGP_CUDA(cudaGetLastError());
    }
    cur = 1 - cur;
  }
  Orders o;
  for (int d = 0; d < 3; d++) o.o[d] = ord[d][cur];
  GGP_CUDA(allow_dyn_smem(tree_sub_kernel, sizeof(SubTree)));
  tree_sub_kernel<<<(unsigned)(int64_t(1) << l0), kSub, sizeof(SubTree), s>>>(
      pts, N, l0, levels, rule, o, start, (int32_t*)flags, tree_point, split_dim, inorder,
      node_at_inorder, box);
  GGP_CUDA(cudaGetLastError());
  return GRAPHGP_OK;
}

}  // namespace ggp
