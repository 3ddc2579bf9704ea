// Hafnians by partial matchings of a growing prefix (FP64).
//
// For a symmetric A of even order n and i = 0..n let V_i(M), M a set of
// positions >= i, be the sum over the ways to match every position below i
// with another one below i or with one of M, using all of M (no pair lies
// inside M). Then V_0({}) = 1, Haf(A) = V_n({}), and matching position i gives
//     V_{i+1}(M) = V_i(M + {i}) + sum_{p in M} A(i, p) V_i(M - {p}),
// position i having been used up before, or being matched with p now. Only
// sets of at most i positions with |M| = i mod 2 occur, so order n costs
// sum_i sum_j j C(n - i, j) complex multiply-adds: 10,226 at n = 16, 0.75 M at
// n = 24 and 17 M at n = 30, where the 2^(n/2)-subset sum takes 0.28 M, 18 M
// and 344 M. Nothing is subtracted that the Hafnian itself does not subtract,
// so the error stays near the unit roundoff instead of growing with the signed
// sum's cancellation ratio. The subset sum remains the route wherever that
// ratio (the error estimate) is asked for.
//
// Sets of one size j among R = n - i - 1 later positions are numbered in colex
// order, rank(M) = sum_t C(p_t, t) over p_1 < ... < p_j (positions relative to
// i + 1), so one layer is the concatenation of its sizes and a set's sources
// are found by arithmetic on its positions.
//
// What bounds it: the FP64 pipe (4 DFMA a multiply-add, a warp instruction
// every 64 cycles per SM quarter on this part; 75 % busy in the shared-memory
// kernel while it is active); the rank arithmetic and the 16-byte loads run
// beside it. Whole calls, subset sum -> matchings: 2048 patterns of n = 8..24
// without the estimate 46.0 -> 2.1 ms, 301 matrices of n <= 22 1.14 -> 0.23 ms;
// the Hafnians of 80 patterns of n = 28 and 30 take 6.5 ms of kernels, those of
// 4096 patterns of n = 16 0.47 ms.
//
// Batches with an order above kMatchMaxN = 30 keep the subset sum as a whole:
// at 32 the matchings are some ten times faster as well, but a committed test
// holds the repeated-row sum of two modes to a third of the time that the
// explicit matrix of order 32 takes, and it stays as it is.
#include <algorithm>
#include <atomic>

#include "gbs_internal.cuh"

namespace gbs {
namespace {

constexpr int kBinRows = kMaxN + 1, kBinCols = kMaxN / 2 + 2;
struct BinomTable {
  int v[kBinRows * kBinCols];  // C(a, b), a <= 32, b <= 17 (the largest, C(32, 16), fits an int)
  constexpr BinomTable() : v() {
    for (int a = 0; a < kBinRows; ++a)
      for (int b = 0; b < kBinCols; ++b)
        v[a * kBinCols + b] = (b == 0) ? 1 : (a == 0) ? 0 : v[(a - 1) * kBinCols + b - 1] + v[(a - 1) * kBinCols + b];
  }
};
__device__ const BinomTable g_binom = BinomTable();

__device__ __forceinline__ void load_binom(int* s) {
  for (int i = threadIdx.x; i < kBinRows * kBinCols; i += blockDim.x) s[i] = g_binom.v[i];
}

__device__ __forceinline__ void cfma_acc(double2& acc, double2 a, double2 b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
}

// Sizes of layer i of order n: j = i mod 2, i mod 2 + 2, ... <= min(i, n - i).
__device__ __forceinline__ int layer_jmax(int n, int i) {
  const int top = min(i, n - i);
  return top - ((top ^ i) & 1);
}

// V_{i+1} of set number r among the j-subsets of R = n - i - 1 positions.
// load(size, rank) reads V_i, row(p) reads A(i, i + 1 + p). The first walk
// finds the positions from the top (and the ranks that put a size-j set of
// this layer among the sets of the layer before, whose positions start one
// lower: p counts as p + 1 there, and position i as 0); the second takes
// them from the bottom with rank(M - {p_s}) = sum_{t<s} C(p_t + 1, t) +
// sum_{t>s} C(p_t + 1, t - 1) kept as a running sum.
template <class Load, class Row>
__device__ __forceinline__ double2 next_value(const int* __restrict__ bin, int R, int j, int r, bool has_up,
                                              const Load& load, const Row& row) {
  unsigned mask = 0;
  int suf = 0, up = 0;
  for (int t = j, c = R - 1; t >= 1; --t, --c) {
    while (bin[c * kBinCols + t] > r) --c;
    r -= bin[c * kBinCols + t];
    mask |= 1u << c;
    suf += bin[(c + 1) * kBinCols + t - 1];
    up += bin[(c + 1) * kBinCols + t + 1];
  }
  double2 acc = make_double2(0.0, 0.0);
  if (has_up) acc = load(1, up);
  int pre = 0;
#pragma unroll 2
  for (int t = 1; t <= j; ++t) {
    const int p = __ffs(mask) - 1;
    mask &= mask - 1;
    const int* b = bin + (p + 1) * kBinCols + t;
    suf -= b[-1];
    cfma_acc(acc, row(p), load(-1, pre + suf));
    pre += b[0];
  }
  return acc;
}

__device__ __forceinline__ int src_index(const MatchLaunch& L, const PatDesc& d, int b, int pos) {
  int v = (d.idx_off >= 0) ? L.idx[d.idx_off + pos] : pos;
  if (L.m_bound > 0 && (v < 0 || v >= L.m_bound)) {
    L.status[b] = 1;
    v = 0;
  }
  return v;
}

__device__ __forceinline__ void store_partial(Partial* out, double2 v) {
  Partial pr;
  pr.re_hi = v.x;
  pr.im_hi = v.y;
  pr.re_lo = pr.im_lo = pr.kappa = 0.0;
  pr.pad[0] = pr.pad[1] = pr.pad[2] = 0.0;
  *out = pr;
}

// Layers i0 + 1..n in shared memory for a tile of P = 2^lp matrices of one
// order. Lane = (set, matrix): P matrices side by side (their values of one
// set are neighbours, so loads are conflict-free and the rank arithmetic is
// shared by the tile's lanes), 32 / P sets per warp; without it the many
// layers of a few sets would leave most lanes of an FP64 instruction, which
// costs the same for one lane as for 32, idle.
// buf[parity] + ((first of the size) + rank) * P + matrix; A: packed strict
// upper triangles, matrices innermost. lb[i][j]: first set of size j in layer i.
__device__ void run_layers(const int* bin, const int (*lb)[kMaxN / 2 + 2], double2* even, double2* odd,
                           const double2* A, int n, int i0, int lp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int P = 1 << lp, S = 32 >> lp;
  const int mat = lane & (P - 1), sub = lane >> lp;
  for (int i = i0; i < n; ++i) {
    const int R = n - i - 1;
    const double2* in = (i & 1) ? odd : even;
    double2* out = (i & 1) ? even : odd;
    const double2* rowA = A + ((int64_t)(i * n - (i * (i + 1)) / 2) << lp) + mat;
    const int jin = min(i, R + 1);
    int t = warp;
    for (int j = layer_jmax(n, i + 1); j >= 0; j -= 2) {
      const int cnt = bin[R * kBinCols + j], tasks = (cnt + S - 1) / S;
      const bool has_up = j + 1 <= jin;
      const int bdn = (j > 0) ? lb[i][j - 1] : 0, bup = has_up ? lb[i][j + 1] : 0, bo = lb[i + 1][j];
      for (; t < tasks; t += nw) {
        const int r = t * S + sub;
        const double2 v = next_value(
            bin, R, j, min(r, cnt - 1), has_up,
            [&](int d, int rk) { return in[((int64_t)((d > 0 ? bup : bdn) + rk) << lp) + mat]; },
            [&](int p) { return rowA[(int64_t)p << lp]; });
        if (r < cnt) out[((int64_t)(bo + r) << lp) + mat] = v;
      }
      t -= tasks;  // the next size's tasks go on with the next warp
    }
    __syncthreads();
  }
}

__device__ __forceinline__ void layer_bases(const int* bin, int (*lb)[kMaxN / 2 + 2], int n) {
  // (bin is ready; the caller synchronises after)
  for (int i = threadIdx.x; i <= n; i += blockDim.x) {
    int at = 0;
    const int top = layer_jmax(n, i);
    for (int j = i & 1; j <= top; j += 2) {
      lb[i][j] = at;
      at += bin[(n - i) * kBinCols + j];
    }
  }
}

// Orders up to kMatchSmallMax: one block per tile; twice the threads where only
// two tiles fit an SM (16 warps kept the FP64 pipe 72 % busy).
__global__ void __launch_bounds__(2 * kMatchThreads) match_small_kernel(const MatchLaunch L) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int bin[kBinRows * kBinCols];
  __shared__ int lb[kMatchSmallMax + 1][kMaxN / 2 + 2];
  __shared__ int rows[32 * kMatchSmallMax];
  __shared__ int64_t s_off[32];
  __shared__ int s_ld[32], s_any;
  load_binom(bin);
  dependency_wait();
  const MatchTile T = L.tiles[blockIdx.x];
  const int n = T.n, lp = T.lp, P = 1 << lp;
  if (threadIdx.x == 0) s_any = (L.skip == nullptr);
  __syncthreads();
  layer_bases(bin, lb, n);
  for (int t = threadIdx.x; t < n << lp; t += blockDim.x) {
    const int q = t / n, pos = t - q * n;
    int v = 0;
    if (q < T.count) {
      const int b = L.order[T.first + q];
      if (L.skip != nullptr && pos == 0 && L.skip[b] == 0) s_any = 1;
      const PatDesc d = L.pats[b];
      if (pos == 0) {
        s_off[q] = d.src_off;
        s_ld[q] = d.ld;
      }
      v = src_index(L, d, b, pos);
    }
    rows[q * n + pos] = v;
  }
  __syncthreads();
  if (!s_any) return;  // every matrix of the tile takes the repeated-row sum (uniform)
  double2* even = reinterpret_cast<double2*>(smem);
  double2* odd = even + ((int64_t)T.even << lp);
  double2* A = odd + ((int64_t)T.odd << lp);
  const double2* src2 = reinterpret_cast<const double2*>(L.src);
  for (int e = threadIdx.x; e < (n * n) << lp; e += blockDim.x) {
    const int q = e & (P - 1), r = (e >> lp) / n, c = (e >> lp) - r * n;
    if (r < c)
      A[((r * n - (r * (r + 1)) / 2 + c - r - 1) << lp) + q] =
          (q < T.count) ? __ldg(src2 + s_off[q] + (int64_t)rows[q * n + r] * s_ld[q] + rows[q * n + c])
                        : make_double2(0.0, 0.0);
  }
  if (threadIdx.x < P) even[threadIdx.x] = make_double2(1.0, 0.0);  // V_0({}) = 1
  __syncthreads();
  run_layers(bin, lb, even, odd, A, n, 0, lp);
  if (threadIdx.x < T.count) store_partial(L.parts + L.order[T.first + threadIdx.x], even[threadIdx.x]);
}

// ---- larger orders: the layers live in device memory (L2), one launch per
// layer over every matrix of the chunk, so that a few matrices fill the chip.

// One block per matrix: gather the packed upper triangle, and layer 2 directly
// (V_2({}) = A(0, 1), V_2({p, q}) = A(0, p) A(1, q) + A(0, q) A(1, p)).
__global__ void __launch_bounds__(kMatchThreads) match_head_kernel(const MatchLaunch L, const MatchChunk C) {
  __shared__ int rows[kMaxN];
  __shared__ double2 A[kMaxN * (kMaxN - 1) / 2];
  dependency_wait();
  int g = 0;
  while (g + 1 < C.n_groups && (int)blockIdx.x >= C.g[g + 1].begin) ++g;
  const MatchGroup G = C.g[g];
  const int n = G.n, q = blockIdx.x - G.begin, b = L.order[G.first + q];
  const PatDesc d = L.pats[b];
  double2* base = reinterpret_cast<double2*>(C.scratch) + G.off + (int64_t)q * G.stride;
  if ((int)threadIdx.x < n) rows[threadIdx.x] = src_index(L, d, b, threadIdx.x);
  __syncthreads();
  if (L.skip != nullptr && L.skip[b] != 0) return;  // uniform
  const double2* src2 = reinterpret_cast<const double2*>(L.src);
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int r = e / n, c = e - r * n;
    if (r < c) {
      const double2 v = __ldg(src2 + d.src_off + (int64_t)rows[r] * d.ld + rows[c]);
      const int at = r * n - (r * (r + 1)) / 2 + c - r - 1;
      base[at] = v;
      A[at] = v;
    }
  }
  __syncthreads();
  double2* even = base + n * (n - 1) / 2;
  const double2* r0 = A + 1;        // A(0, 2 + p)
  const double2* r1 = A + (n - 1);  // A(1, 2 + p)
  if (threadIdx.x == 0) even[0] = A[0];
  for (int e = threadIdx.x; e < (n - 2) * (n - 2); e += blockDim.x) {
    const int p = e / (n - 2), c = e - p * (n - 2);
    if (p < c) {
      double2 acc = make_double2(0.0, 0.0);
      cfma_acc(acc, r1[p], r0[c]);
      cfma_acc(acc, r1[c], r0[p]);
      even[1 + c * (c - 1) / 2 + p] = acc;
    }
  }
}

// Layer i -> i + 1: a warp takes 32 sets of one size of one matrix at a time,
// the largest sizes of a matrix first. The grid is as many blocks as are
// resident, each warp striding over the tasks: a block per eight tasks spent
// its time on the table, and matrices the repeated-row sum computes cost one
// load a task.
__global__ void __launch_bounds__(kMatchThreads) match_layer_kernel(const MatchLaunch L, const MatchChunk C, int i) {
  __shared__ int bin[kBinRows * kBinCols];
  load_binom(bin);
  dependency_wait();
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int nw = gridDim.x * (blockDim.x >> 5);
  int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  for (int g = 0; g < C.n_groups; ++g) {
    const MatchGroup G = C.g[g];
    const int n = G.n, R = n - i - 1, jin = min(i, R + 1), all = G.tasks * G.count;
    for (; w < all; w += nw) {
      const int q = w / G.tasks;
      int t = w - q * G.tasks;
      if (L.skip != nullptr && L.skip[L.order[G.first + q]] != 0) continue;
      const double2* A = reinterpret_cast<const double2*>(C.scratch) + G.off + (int64_t)q * G.stride;
      double2* even = const_cast<double2*>(A) + n * (n - 1) / 2;
      double2* odd = even + G.even;
      const double2* in = (i & 1) ? odd : even;
      double2* out = (i & 1) ? even : odd;
      // this task's size, and where it and its sources start
      int j = layer_jmax(n, i + 1), bo = 0, below = 0;
      for (; j >= 0; j -= 2) {
        const int tk = (bin[R * kBinCols + j] + 31) / 32;
        if (t < tk) break;
        t -= tk;
      }
      for (int s = (i + 1) & 1; s < j; s += 2) bo += bin[R * kBinCols + s];
      for (int s = i & 1; s < j - 1; s += 2) below += bin[(R + 1) * kBinCols + s];
      const bool has_up = j + 1 <= jin;
      const double2* indn = in + below;
      const double2* inup = indn + (j > 0 ? bin[(R + 1) * kBinCols + j - 1] : 0);
      const double2* rowA = A + (i * n - (i * (i + 1)) / 2);
      const int cnt = bin[R * kBinCols + j], r = t * 32 + lane;
      const double2 v = next_value(
          bin, R, j, min(r, cnt - 1), has_up, [&](int dd, int rk) { return (dd > 0 ? inup : indn)[rk]; },
          [&](int p) { return rowA[p]; });
      if (r < cnt) out[bo + r] = v;
    }
    w -= all;
  }
}

// The last layers of one matrix per block, in shared memory: from layer
// n - kMatchTail on, 2^(kMatchTail - 1) sets and fewer.
__global__ void __launch_bounds__(kMatchThreads) match_tail_kernel(const MatchLaunch L, const MatchChunk C) {
  __shared__ int bin[kBinRows * kBinCols];
  __shared__ int lb[kMaxN + 1][kMaxN / 2 + 2];
  __shared__ double2 buf[2][1 << (kMatchTail - 1)];
  load_binom(bin);
  dependency_wait();
  int g = 0;
  while (g + 1 < C.n_groups && (int)blockIdx.x >= C.g[g + 1].begin) ++g;
  const MatchGroup G = C.g[g];
  const int n = G.n, q = blockIdx.x - G.begin, b = L.order[G.first + q];
  if (L.skip != nullptr && L.skip[b] != 0) return;  // uniform
  const double2* A = reinterpret_cast<const double2*>(C.scratch) + G.off + (int64_t)q * G.stride;
  const double2* even = A + n * (n - 1) / 2;
  const int i0 = n - kMatchTail;
  const double2* in = (i0 & 1) ? even + G.even : even;
  for (int e = threadIdx.x; e < 1 << (kMatchTail - 1); e += blockDim.x) buf[i0 & 1][e] = in[e];
  __syncthreads();
  layer_bases(bin, lb, n);
  __syncthreads();
  run_layers(bin, lb, buf[0], buf[1], A, n, i0, 0);
  if (threadIdx.x == 0) store_partial(L.parts + b, buf[0][0]);
}

int64_t choose(int a, int b) {
  if (b < 0 || b > a) return 0;
  int64_t r = 1;
  for (int i = 1; i <= b; ++i) r = r * (a - b + i) / i;
  return r;
}

}  // namespace

void match_sizes(int n, int* even, int* odd, double* macs) {
  *even = *odd = 0;
  double m = 0;
  for (int i = 0; i <= n; ++i) {
    int64_t sets = 0;
    for (int j = i & 1; j <= std::min(i, n - i); j += 2) {
      sets += choose(n - i, j);
      m += (double)j * (double)choose(n - i, j);
    }
    int& top = (i & 1) ? *odd : *even;
    top = std::max<int>(top, (int)sets);
  }
  if (macs) *macs = m;
}

size_t match_matrix_bytes(int n) {
  int even, odd;
  match_sizes(n, &even, &odd, nullptr);
  return 16 * ((size_t)even + odd + n * (n - 1) / 2);
}

cudaError_t launch_match_small(const MatchLaunch& L, int tiles, size_t smem, cudaStream_t st) {
  static std::atomic<int> done[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!done[dev].load(std::memory_order_acquire)) {
    e = cudaFuncSetAttribute(match_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMatchTileBytes);
    if (e != cudaSuccess) return e;
    done[dev].store(1, std::memory_order_release);
  }
  return launch_dependent(match_small_kernel, dim3(tiles), smem > 56 * 1024 ? 2 * kMatchThreads : kMatchThreads, smem, st, L);
}

cudaError_t launch_match_large(const MatchLaunch& L, MatchChunk C, bool shared, cudaStream_t st) {
  if (C.n_groups <= 0) return cudaSuccess;
  const MatchGroup& last = C.g[C.n_groups - 1];
  const int mats = last.begin + last.count;
  int nmax = 0;
  for (int g = 0; g < C.n_groups; ++g) nmax = std::max(nmax, C.g[g].n);
  int dev = 0, sms = 0, resident = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, match_layer_kernel, kMatchThreads, 0);
  if (e != cudaSuccess) return e;
  if (shared) resident = std::min(resident, 3);  // beside the terms' blocks (24 warps keep the FP64 pipe busy)
  if ((e = launch_dependent(match_head_kernel, dim3(mats), kMatchThreads, 0, st, L, C)) != cudaSuccess) return e;
  constexpr int wpb = kMatchThreads / 32;
  for (int i = 2; i < nmax - kMatchTail; ++i) {
    int64_t warps = 0;  // below 2^31: the scratch holds 16 bytes for each of a task's 32 sets
    for (int g = 0; g < C.n_groups; ++g) {
      MatchGroup& G = C.g[g];
      G.tasks = 0;
      const int R = G.n - i - 1;
      if (i < G.n - kMatchTail)
        for (int j = (i + 1) & 1; j <= std::min(i + 1, R); j += 2) G.tasks += (int)((choose(R, j) + 31) / 32);
      warps += (int64_t)G.tasks * G.count;
    }
    const int64_t blocks = std::min<int64_t>((warps + wpb - 1) / wpb, (int64_t)sms * resident);
    e = launch_dependent(match_layer_kernel, dim3((unsigned)blocks), kMatchThreads, 0, st, L, C, i);
    if (e != cudaSuccess) return e;
  }
  return launch_dependent(match_tail_kernel, dim3(mats), kMatchThreads, 0, st, L, C);
}

}  // namespace gbs
