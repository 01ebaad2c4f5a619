// The dense initial block (the dense initial batch of Alg. 1; Sec. 2.2 "Batch
// construction"): L0 = chol(K_00 + nugget I), L0^-1, sigma_i = L0_ii and
// sum log L0_ii^2.
//
// One cooperative launch: a right-looking Cholesky over 32 x 32 tiles, the
// blocks on a px x py grid owning tiles (I, K), I = a mod px, K = b mod py.
// Per panel J there is one grid barrier: every block factors the diagonal
// tile itself (one warp, lane = row, the row in registers), solves the panel
// rows of the tile rows it needs (one warp each, the same routine with the
// pivots given) and applies them to its tiles, whose accumulators stay in L2.
// Doing the diagonal tile and the solves redundantly costs less than the two
// further barriers that sharing them would take.  The inverse follows in the
// same launch, rows or columns of L0^-1 being independent of each other.
// Bound by latency (32 dependent pivots per panel, a barrier each), not by
// arithmetic; the former one-block kernels took 0.74 ms at n0 = 256 and about
// 105 ms at n0 = 1000, where one SM had to move n0^3 / 3 operands.
//
// The order of every FP32 sum is that of a left-looking evaluation with
// separate partial sums, and is kept across panels because a tile's partial
// sums are accumulated in ascending m:
//   n0 <= 320: t_rj = K_rj - ((s_0 + s_1) + (s_2 + s_3)), s_p over m = p mod 4;
//     W_rj = -(1 / L_jj) of the same four sums of W_rm L_mj over m = j + 1 + p
//     mod 4, last column first (rows of W are independent);
//   n0 > 320:  t_rj = t_0 + t_1, t_0 from K_rj over the even m, t_1 over the
//     odd m; W_ij = -(sum_m L_im W_mj) / L_ii in one sum (columns independent).
// Pivots below 1e-7 K_00 are raised to that floor and counted.
//
// The FP32 block's error is estimated like a conditional's (rescue.cuh): every
// dense row is a conditional on all earlier dense points, with K_jj = K_00 for
// every j, so est = 2^-24 (K_00 / p_min)^2 from the smallest FP32 pivot p_min.
// When the estimate exceeds the kernel's rescue_tol or a pivot was floored, a
// second launch of the same kernel in FP64 (distances, tiles, inverse)
// replaces L0 and L0^-1, rounded to FP32; else it only adds the FP32 block's
// log-determinant and floor count to the factor's.
#include <algorithm>

#include "pointfactor.cuh"
#include "sweepsync.cuh"

namespace ggp {
namespace {

constexpr int kT = 32;            // tile edge
constexpr int kDenseThreads = 256;
constexpr int kDenseSplitMax = 320;  // largest n0 of the four-sum order
// Polls that a wait for the other blocks' panel gets beside the graph's max_spin: a
// panel is under 1 ms of work at any n0, a poll about 0.7 us.  A caller may bound
// the waits of the sweeps tightly; the factor, which needs no such bound, has to
// succeed all the same.
constexpr int64_t kDensePolls = 1 << 20;

struct DenseCheck {
  double logdet;           // sum log L0_ii^2 of the FP32 block
  unsigned long long bad;  // floored pivots
  int min_piv;             // smallest accepted pivot (FP32 bits; positive)
};

struct DenseArgs {
  const float4* xs;
  int n0, nb;       // points, tiles per side
  int px, py;       // block grid
  KernF kf;
  void* acc;        // accumulators, [tile][plane][column][row]
  void* LT;         // L0 transposed, n0 x n0
  float* L0;
  float* L0inv;
  float* sigma;
  DenseCheck* chk;
  double* logdet;
  unsigned long long* not_pd;
  LevelBarrier lb;
};

// T: FP32 or FP64; NP: partial sums.  NP = 4 keeps K beside the sums.
template <class T, int NP>
struct DenseForm {
  static constexpr int planes = NP == 4 ? 5 : NP;
  // t of an element from its planes
  static __device__ __forceinline__ T value(const T (&p)[planes]) {
    if constexpr (NP == 4) return p[4] - ((p[0] + p[1]) + (p[2] + p[3]));
    else if constexpr (NP == 2) return p[0] + p[1];
    else return p[0];
  }
  static __device__ __forceinline__ T add(T acc, T x, T y) {
    return NP == 4 ? fma(x, y, acc) : fma(-x, y, acc);
  }
};

template <class T, int KT>
__device__ __forceinline__ T dense_entry(const DenseArgs& d, int i, int j) {
  if (i >= d.n0 || j >= d.n0) return T(0);
  if constexpr (sizeof(T) == 4) {
    if (i == j) return d.kf.s2 + d.kf.nug;
    return kappa_d2<KT>(d.kf, sqdist(d.xs[i], d.xs[j]));
  } else {
    if (i == j) return d.kf.s2d + d.kf.nugd;
    return kappa64<KT>(d.kf, dist64(d.xs[i], d.xs[j]));
  }
}

__device__ __forceinline__ float droot(float x) { return sqrt_newton(x); }
__device__ __forceinline__ double droot(double x) { return sqrt(x); }
__device__ __forceinline__ float drcp(float x) { return rcp_newton(x); }
__device__ __forceinline__ double drcp(double x) { return x; }
// t / L_jj: FP32 by the reciprocal, FP64 by division (`iv` is L_jj itself)
__device__ __forceinline__ float scaled(float t, float iv) { return t * iv; }
__device__ __forceinline__ double scaled(double t, double ljj) { return t / ljj; }

// One warp, lane = row of the tile at `tile` (planes of [column][row]): the
// row's 32 columns of L against the diagonal tile's.  DIAG: the tile is the
// diagonal one; pivots are found (floored, counted in `bad`, the smallest
// accepted one in `pmin`) and D[j][r] and inv[j] (drcp of L_jj) are written; else they are read.
// The row's entries are left in out[column][row] (DIAG: D itself) and, when lt
// is given, in L0's transpose (lt: the row's entry of the tile's first column,
// n0 apart; null for rows that do not exist).  `cols`: columns that exist; fewer than
// the tile's only on the last diagonal tile, which has a copy of this that stops
// there (SHORT: a test per column makes every panel 3 % slower).
template <class T, int NP, bool DIAG, bool SHORT = false>
__device__ __noinline__ void tile_rows(const T* tile, T* D, T* inv, T* out, T* lt, int n0, int cols,
                                       T fl, unsigned& bad, T& pmin) {
  using F = DenseForm<T, NP>;
  const int r = threadIdx.x & 31;
  T a[NP][kT], m0[NP == 4 ? kT : 1];
#pragma unroll
  for (int c = 0; c < kT; c++) {
#pragma unroll
    for (int p = 0; p < NP; p++) a[p][c] = __ldcg(tile + (p * kT + c) * kT + r);
    if constexpr (NP == 4) m0[c] = __ldcg(tile + (4 * kT + c) * kT + r);
  }
#pragma unroll
  for (int j = 0; j < kT; j++) {
    if (SHORT && j >= cols) {
      D[j * kT + r] = T(0);
      if (r == j) inv[j] = T(1);
      continue;
    }
    T pl[F::planes];
#pragma unroll
    for (int p = 0; p < NP; p++) pl[p] = a[p][j];
    if constexpr (NP == 4) pl[4] = m0[j];
    const T t = F::value(pl);
    T l;
    if (DIAG) {
      T piv = __shfl_sync(0xffffffffu, t, j);
      if (!(piv > fl)) {
        piv = fl;
        bad++;
      } else {
        pmin = piv < pmin ? piv : pmin;
      }
      const T ljj = droot(piv);
      const T iv = drcp(ljj);
      l = r > j ? scaled(t, iv) : (r == j ? ljj : T(0));
      D[j * kT + r] = l;
      if (r == j) inv[j] = iv;
      __syncwarp();
    } else {
      l = scaled(t, inv[j]);
      out[j * kT + r] = l;
    }
    if (lt) lt[(int64_t)j * n0] = l;
#pragma unroll
    for (int c = j + 1; c < kT; c++) a[j % NP][c] = F::add(a[j % NP][c], l, D[j * kT + c]);
  }
}

// L0 row-major, upper part zero, from its transpose: the block's share of the
// nb x nb tiles through shared memory (tr: kT x (kT + 1)).
template <class T>
__device__ __forceinline__ void write_L0(const DenseArgs& d, const T* LT, float* tr) {
  const int n0 = d.n0, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int e = blockIdx.x; e < d.nb * d.nb; e += gridDim.x) {
    const int I = e / d.nb, K = e % d.nb;
    if (K <= I)
      for (int c = warp; c < kT; c += kDenseThreads / 32) {
        const int row = I * kT + lane, col = K * kT + c;
        tr[c * (kT + 1) + lane] =
            row < n0 && col <= row ? (float)LT[(int64_t)col * n0 + row] : 0.0f;
      }
    __syncthreads();
    for (int r = warp; r < kT; r += kDenseThreads / 32) {
      const int row = I * kT + r, col = K * kT + lane;
      if (row < n0 && col < n0)
        d.L0[(int64_t)row * n0 + col] = K <= I ? tr[lane * (kT + 1) + r] : 0.0f;
    }
    __syncthreads();
  }
}

// Rows of L^-1, four lanes per row, last column first (n0 <= 320, FP32).  Lane
// rho holds the entries m = rho mod 4 of the row and of the columns of L, in
// shared memory, four of them per load (column j: the groups of 32 rows from
// that of row j on, [rho][8] each; the row likewise).  At step j it is the sum
// p = (rho - j - 1) mod 4 of the order above; entries of the row that are not
// formed yet or do not exist are zero and drop out.  Bound by the chain of a
// step's additions: 45 us at n0 = 256 (150 us with one entry per load).
constexpr int kInvG = 32;
__device__ __forceinline__ int inv_col(int j, int n0) {  // offset of column j
  const int G = (n0 + kInvG - 1) / kInvG, g = j / kInvG;  // groups before: sum of (G - g') kInvG columns
  return kInvG * (kInvG * (g * G - g * (g - 1) / 2) + (j - g * kInvG) * (G - g));
}
__device__ __forceinline__ int inv_slot(int m) {  // place of entry m in its group
  return m / kInvG * kInvG + (m & 3) * (kInvG / 4) + m % kInvG / 4;
}

__device__ __forceinline__ void inverse_rows(const DenseArgs& d, const float* Ls, const float* dinv,
                                             float* W, int ld, int first, int rows) {
  const int lane = threadIdx.x & 31, rho = lane & 3, n0 = d.n0;
  const int q = lane >> 2 < rows ? lane >> 2 : 0, r = first + q;
  float* Wr = W + q * ld;
  for (int e = lane; e < rows * ld; e += 32) W[e] = 0.0f;
  __syncwarp();
  const int top = min(first + rows - 1, n0 - 1);
  if (r < n0) Wr[inv_slot(r)] = dinv[r];
  __syncwarp();
  const int gtop = top / kInvG;
  for (int j = top - 1; j >= 0; j--) {
    const int g0 = j / kInvG;
    const float* Lj = Ls + inv_col(j, n0) - g0 * kInvG + rho * (kInvG / 4);
    const float* Wl = Wr + rho * (kInvG / 4);
    float acc = 0.0f;
#pragma unroll 2
    for (int g = g0; g <= gtop; g++) {
      const float4 x0 = *reinterpret_cast<const float4*>(Lj + g * kInvG);
      const float4 x1 = *reinterpret_cast<const float4*>(Lj + g * kInvG + 4);
      const float4 w0 = *reinterpret_cast<const float4*>(Wl + g * kInvG);
      const float4 w1 = *reinterpret_cast<const float4*>(Wl + g * kInvG + 4);
      acc = fmaf(w0.x, x0.x, acc);
      acc = fmaf(w0.y, x0.y, acc);
      acc = fmaf(w0.z, x0.z, acc);
      acc = fmaf(w0.w, x0.w, acc);
      acc = fmaf(w1.x, x1.x, acc);
      acc = fmaf(w1.y, x1.y, acc);
      acc = fmaf(w1.z, x1.z, acc);
      acc = fmaf(w1.w, x1.w, acc);
    }
    const int p = (rho - j - 1) & 3;
    const int base = lane & ~3;
    acc += __shfl_sync(0xffffffffu, acc, base + (((p ^ 1) + j + 1) & 3));
    acc += __shfl_sync(0xffffffffu, acc, base + (((p ^ 2) + j + 1) & 3));
    if (rho == (j & 3) && j < r && r < n0) Wr[inv_slot(j)] = -dinv[j] * acc;
    __syncwarp();
  }
  for (int e = lane; e < rows * n0; e += 32) {
    const int row = first + e / n0, c = e % n0;
    if (row < n0) d.L0inv[(int64_t)row * n0 + c] = c <= row ? W[(e / n0) * ld + inv_slot(c)] : 0.0f;
  }
  __syncwarp();
}

// Stride of the rows of W (entries of all groups, then a skew of four banks)
// and rows per warp: at n0 > 288 the columns of L leave room for four.
__host__ __device__ constexpr int inverse_ld(int n0) { return (n0 + kInvG - 1) / kInvG * kInvG + 4; }
__host__ __device__ constexpr int inverse_rows_per_warp(int n0) { return n0 > 288 ? 4 : 8; }

// CW columns of L^-1 by forward substitution, the block's threads holding the
// sums of all rows: row m is finished (one row per step), then added to the
// rows below it, in ascending m.
template <class T, int CW>
__device__ __forceinline__ void inverse_columns(const DenseArgs& d, const T* LT, T* ws, int c0) {
  constexpr int Q = 2048 / kDenseThreads;
  const int n0 = d.n0, tid = threadIdx.x;
  for (int e = tid; e < c0 * CW; e += kDenseThreads) {
    const int c = c0 + e % CW;
    if (c < n0) d.L0inv[(int64_t)(e / CW) * n0 + c] = 0.0f;
  }
  T t[Q][CW], l[Q];
#pragma unroll
  for (int q = 0; q < Q; q++) {
#pragma unroll
    for (int c = 0; c < CW; c++) t[q][c] = T(0);
    const int i = q * kDenseThreads + tid;
    l[q] = i < n0 ? LT[(int64_t)c0 * n0 + i] : T(0);
  }
  for (int m = c0; m < n0; m++) {
    T* w = ws + (m & 1) * 2 * CW;
    // row m's sums to its warp, which divides them
    if ((m % kDenseThreads) >> 5 == tid >> 5) {
      const int q0 = m / kDenseThreads;
#pragma unroll
      for (int q = 0; q < Q; q++)
        if (q == q0 && tid == m % kDenseThreads) {
#pragma unroll
          for (int c = 0; c < CW; c++) w[CW + c] = t[q][c];
          ws[4 * CW] = l[q];
        }
      __syncwarp();
      const int c = tid & 31;
      if (c < CW && c0 + c < n0) {
        const T lmm = ws[4 * CW];
        const T v = c0 + c < m ? -w[CW + c] / lmm : (c0 + c == m ? T(1) / lmm : T(0));
        w[c] = v;
        d.L0inv[(int64_t)m * n0 + c0 + c] = (float)v;
      } else if (c < CW) {
        w[c] = T(0);
      }
    }
    __syncthreads();
    T x[CW];
#pragma unroll
    for (int c = 0; c < CW; c++) x[c] = w[c];
#pragma unroll
    for (int q = 0; q < Q; q++) {
      const int i = q * kDenseThreads + tid;
      if (q * kDenseThreads < n0 && (q + 1) * kDenseThreads > m + 1) {
        const T lq = l[q];
        if (i < n0 && m + 1 < n0) l[q] = LT[(int64_t)(m + 1) * n0 + i];
#pragma unroll
        for (int c = 0; c < CW; c++) t[q][c] = fma(lq, x[c], t[q][c]);
      }
    }
  }
  __syncthreads();
}

template <class T, int NP, int KT>
__global__ void __launch_bounds__(kDenseThreads, 1) dense_block_kernel(DenseArgs d) {
  using F = DenseForm<T, NP>;
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ int s_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if constexpr (sizeof(T) == 8) {  // FP64: only when the FP32 block is not good enough
    const float r32 = (d.kf.s2 + d.kf.nug) / __int_as_float(d.chk->min_piv);
    if (d.chk->bad == 0 && r32 * r32 <= d.kf.resc_T) {
      if (blockIdx.x == 0 && tid == 0) atomicAdd(d.logdet, d.chk->logdet);
      return;
    }
  }
  const int nb = d.nb, px = d.px, py = d.py;
  // block -> (a, b): the lower triangle of the block grid when a tile row has
  // a block of its own, else the whole grid
  int a, b;
  if (px == nb) {
    a = 0;
    int base = 0;
    while (base + a + 1 <= (int)blockIdx.x) base += ++a;
    b = blockIdx.x - base;
  } else {
    a = blockIdx.x / py;
    b = blockIdx.x % py;
  }
  T* acc = static_cast<T*>(d.acc);
  T* LT = static_cast<T*>(d.LT);
  constexpr int64_t kTileElems = (int64_t)F::planes * kT * kT;
  auto tile = [&](int I, int K) { return acc + ((int64_t)I * (I + 1) / 2 + K) * kTileElems; };
  T* D = reinterpret_cast<T*>(dsm);           // diagonal tile [column][row]
  T* inv = D + kT * kT;                       // [kT]
  const int per = (nb + px - 1) / px;
  T* LI = inv + kT;                           // rows I: [per][column][row]
  T* LK = LI + (int64_t)per * kT * kT;        // rows K: [per][column][row]
  // element pairs of a tile that this thread owns: rows r2, r2 + 1, columns c2, c2 + 1
  const int r2 = 2 * (tid & 15), c2 = 2 * (tid >> 4);
  for (int I = a; I < nb; I += px)
    for (int K = b; K <= I; K += py) {
      T* A = tile(I, K);
      for (int e = 0; e < 4; e++) {
        const int r = r2 + (e & 1), c = c2 + (e >> 1);
        const T v = dense_entry<T, KT>(d, I * kT + r, K * kT + c);
#pragma unroll
        for (int p = 0; p < NP; p++) A[(p * kT + c) * kT + r] = (NP != 4 && p == 0) ? v : T(0);
        if constexpr (NP == 4) A[(4 * kT + c) * kT + r] = v;
      }
    }
  __syncthreads();
  d.lb.arrive(0);
  const T k0 = sizeof(T) == 4 ? T(d.kf.s2 + d.kf.nug) : T(d.kf.s2d + d.kf.nugd);
  const T fl = sizeof(T) == 4 ? T(fmaxf(kPdFloor * (float)k0, kPivotMin)) : T(kPdFloor64 * k0);
  for (int J = 0; J < nb; J++) {
    if (d.lb.wait(J, gridDim.x, &s_flag)) return;
    const int cols = min(kT, d.n0 - J * kT);
    if (warp == 0) {
      unsigned bad = 0;
      T pmin = k0;
      const bool own = a == J % px && b == J % py;  // writes it out
      T* lt = own && lane < cols ? LT + (int64_t)J * kT * d.n0 + J * kT + lane : nullptr;
      if (cols < kT)
        tile_rows<T, NP, true, true>(tile(J, J), D, inv, nullptr, lt, d.n0, cols, fl, bad, pmin);
      else
        tile_rows<T, NP, true>(tile(J, J), D, inv, nullptr, lt, d.n0, cols, fl, bad, pmin);
      __syncwarp();
      if (own) {
        double ls = 0.0;
        if (lane < cols) {
          const float l = (float)D[lane * kT + lane];
          d.sigma[J * kT + lane] = l;
          ls = log((double)l * (double)l);
        }
        for (int o = 16; o; o >>= 1) ls += __shfl_xor_sync(0xffffffffu, ls, o);
        if (lane == 0) {
          if constexpr (sizeof(T) == 4) {
            atomicAdd(&d.chk->logdet, ls);
            if (bad) atomicAdd(&d.chk->bad, (unsigned long long)bad);
            atomicMin(&d.chk->min_piv, __float_as_int((float)pmin));
          } else {
            atomicAdd(d.logdet, ls);
            if (bad) atomicAdd(d.not_pd, (unsigned long long)bad);
          }
        }
      }
    }
    __syncthreads();
    // panel rows: warps take the tile rows I = a mod px, then K = b mod py
    const int qi = J < a ? 0 : (J - a) / px + 1;  // first I = a + qi px > J
    const int qk = J < b ? 0 : (J - b) / py + 1;
    const int ni = (nb - a + px - 1) / px - qi, nk = (nb - b + py - 1) / py - qk;
    for (int w = warp; w < ni + nk; w += kDenseThreads / 32) {
      const bool isI = w < ni;
      const int q = isI ? qi + w : qk + (w - ni);
      const int R = isI ? a + q * px : b + q * py;
      T* out = (isI ? LI : LK) + (int64_t)q * kT * kT;
      unsigned bad = 0;
      T pmin = k0;
      const int row = R * kT + lane;
      tile_rows<T, NP, false>(tile(R, J), D, inv, out,
                              isI && b == J % py && row < d.n0
                                  ? LT + (int64_t)J * kT * d.n0 + row
                                  : nullptr,
                              d.n0, cols, fl, bad, pmin);
    }
    __syncthreads();
    for (int I = a + qi * px, q = qi; I < nb; I += px, q++)
      for (int K = b + qk * py, s = qk; K <= I; K += py, s++) {
        const T* X = LI + (int64_t)q * kT * kT + r2;
        const T* Y = LK + (int64_t)s * kT * kT + c2;
        T* A = tile(I, K);
        T u[NP][4];
#pragma unroll
        for (int p = 0; p < NP; p++)
#pragma unroll
          for (int e = 0; e < 4; e++) u[p][e] = A[(p * kT + c2 + (e >> 1)) * kT + r2 + (e & 1)];
#pragma unroll 8
        for (int m = 0; m < kT; m++) {
          const T x0 = X[m * kT], x1 = X[m * kT + 1], y0 = Y[m * kT], y1 = Y[m * kT + 1];
          u[m % NP][0] = F::add(u[m % NP][0], x0, y0);
          u[m % NP][1] = F::add(u[m % NP][1], x1, y0);
          u[m % NP][2] = F::add(u[m % NP][2], x0, y1);
          u[m % NP][3] = F::add(u[m % NP][3], x1, y1);
        }
#pragma unroll
        for (int p = 0; p < NP; p++)
#pragma unroll
          for (int e = 0; e < 4; e++) A[(p * kT + c2 + (e >> 1)) * kT + r2 + (e & 1)] = u[p][e];
      }
    __syncthreads();
    d.lb.arrive(J + 1);
  }
  if (d.lb.wait(nb, gridDim.x, &s_flag)) return;
  write_L0<T>(d, LT, reinterpret_cast<float*>(dsm));
  if constexpr (sizeof(T) == 4 && NP == 4) {
    // one warp per block takes a few rows at a time; the others help to load
    const int ld = inverse_ld(d.n0), rows = inverse_rows_per_warp(d.n0);
    const int groups = (d.n0 + rows - 1) / rows;
    if ((int)blockIdx.x >= groups) return;
    float* W = reinterpret_cast<float*>(dsm);
    float* dinv = W + rows * ld;
    float* Ls = dinv + ld;
    for (int j = warp; j < d.n0; j += kDenseThreads / 32) {
      const int g0 = j / kInvG * kInvG;
      float* Lj = Ls + inv_col(j, d.n0) - g0;
      for (int m = g0 + lane; m < ld - 4; m += 32)
        Lj[inv_slot(m)] = m > j && m < d.n0 ? LT[(int64_t)j * d.n0 + m] : 0.0f;
      if (lane == 0) dinv[j] = 1.0f / LT[(int64_t)j * d.n0 + j];
    }
    __syncthreads();
    if (warp == 0)
      for (int gr = blockIdx.x; gr < groups; gr += gridDim.x)
        inverse_rows(d, Ls, dinv, W, ld, gr * rows, rows);
  } else {
    constexpr int CW = sizeof(T) == 4 ? 8 : 4;
    for (int c0 = blockIdx.x * CW; c0 < d.n0; c0 += gridDim.x * CW)
      inverse_columns<T, CW>(d, LT, reinterpret_cast<T*>(dsm), c0);
  }
}

// Dynamic shared memory of a launch with `per` tile rows a block and side.
template <class T, int NP>
size_t dense_smem(int n0, int per) {
  size_t b = ((size_t)(1 + 2 * per) * kT * kT + kT) * sizeof(T);
  if (NP == 4) {
    const size_t G = (n0 + kInvG - 1) / kInvG, cols = kInvG * kInvG * G * (G + 1) / 2;
    b = std::max(b, ((inverse_rows_per_warp(n0) + 1) * (size_t)inverse_ld(n0) + cols) * 4);
  }
  return b;
}

template <class T, int NP, int KT>
int launch_dense(DenseArgs d, cudaStream_t s) {
  auto kern = dense_block_kernel<T, NP, KT>;
  // a square block grid, at most one block per SM
  int side = 1;
  while ((side + 1) * (side + 1) <= num_sms()) side++;
  d.px = d.py = std::min(d.nb, side);
  const int grid = d.px == d.nb ? d.nb * (d.nb + 1) / 2 : d.px * d.py;
  const size_t smem = dense_smem<T, NP>(d.n0, (d.nb + d.px - 1) / d.px);
  GGP_CUDA(allow_dyn_smem(kern, smem));
  if (grid == 1) {  // nothing to wait for: a plain launch, which costs less
    kern<<<1, kDenseThreads, smem, s>>>(d);
    GGP_CUDA(cudaGetLastError());
    return GRAPHGP_OK;
  }
  void* args[] = {(void*)&d};
  GGP_CUDA(cudaLaunchCooperativeKernel((const void*)kern, dim3(grid), dim3(kDenseThreads), args,
                                       smem, s));
  return GRAPHGP_OK;
}

template <int KT>
int dense_factor_kt(graphgp_graph_t g, graphgp_factor_t f, const KernF& kf, cudaStream_t s) {
  DenseArgs d{};
  d.xs = g->xs;
  d.n0 = g->n0;
  d.nb = (g->n0 + kT - 1) / kT;
  d.kf = kf;
  d.L0 = f->L0;
  d.L0inv = f->L0inv;
  d.sigma = f->sigma;
  d.logdet = f->logdet;
  d.not_pd = f->not_pd;
  const bool split = g->n0 <= kDenseSplitMax;
  const size_t tiles = (size_t)d.nb * (d.nb + 1) / 2 * kT * kT;
  // accumulators and L0^T of either precision, the check, two sets of counters
  const size_t acc_bytes = tiles * std::max<size_t>(split ? 5 * sizeof(float) : 0, sizeof(double));
  const size_t lt_bytes = (size_t)g->n0 * g->n0 * sizeof(double);
  Scratch sc(s);
  unsigned char* work = nullptr;
  uint32_t* small = nullptr;
  const size_t nsmall = sizeof(DenseCheck) / 4 + 2 * (d.nb + 1);
  GGP_TRY(sc.alloc(&work, acc_bytes + lt_bytes));
  GGP_TRY(sc.alloc(&small, nsmall));
  d.acc = work;
  d.LT = work + acc_bytes;
  d.chk = reinterpret_cast<DenseCheck*>(small);
  GGP_CUDA(cudaMemsetAsync(small, 0, nsmall * 4, s));
  GGP_CUDA(cudaMemsetAsync(&d.chk->min_piv, 0x7f, sizeof(int), s));  // 3.4e38
  d.lb = LevelBarrier{small + sizeof(DenseCheck) / 4, g->err, g->max_spin + kDensePolls};
  if (split)
    GGP_TRY((launch_dense<float, 4, KT>(d, s)));
  else
    GGP_TRY((launch_dense<float, 2, KT>(d, s)));
  d.lb.count += d.nb + 1;
  return launch_dense<double, 1, KT>(d, s);
}

}  // namespace

int dense_factor(graphgp_graph_t g, graphgp_factor_t f, const KernF& kf, int type,
                 cudaStream_t s) {
  switch (type) {
    case GRAPHGP_MATERN12: return dense_factor_kt<GRAPHGP_MATERN12>(g, f, kf, s);
    case GRAPHGP_MATERN32: return dense_factor_kt<GRAPHGP_MATERN32>(g, f, kf, s);
    case GRAPHGP_MATERN52: return dense_factor_kt<GRAPHGP_MATERN52>(g, f, kf, s);
    default: return dense_factor_kt<GRAPHGP_SQEXP>(g, f, kf, s);
  }
}

}  // namespace ggp
