// Marginal probabilities q_n(x_1..x_k) of the position-basis distribution and
// the chain-rule sampler built on them (Sec. 3.3-3.4, Theorem 1, Algorithms 1
// and 2). Identical squeezing only: the theorem collapses the sums over the
// unsampled photons with the unitarity of W = U U^T (Rule 3:
// sum_i W(i, j) conj(W(i, j')) = delta_jj'); for B = U diag(tanh r_i) U^T with
// unequal r_i that sum is (U* diag(tanh^2 r) U^T)_{j'j}, not a multiple of
// delta, so the theorem does not apply (and q_n does not depend on r when the
// r_i are equal).
//
// Theorem 1, as used here (with the index sets of Algorithm 2):
//   q_n(x_1..x_k) = sum_{ja, jb} sum_{s in C([k], ja), s' in C([k], jb)}
//       Haf(W_s) conj(Haf(W_s')) sum_mu F(k, mu, ja, jb) / f_n
//       sum_{A in C([k] \ s, mu), B in C([k] \ s', mu)} Per(S_{A,B})
//       Haf(W_e) conj(Haf(W_e')),   e = [k] \ (s u A), e' = [k] \ (s' u B),
// ja, jb even in [max(0, 2k - n), k], mu in [max(0, 3k - ja - jb - n), k - max(ja, jb)],
// F = (n-k)! C((n-k+mu+m)/2 - 1, k - (ja+jb)/2 + m/2 - 1) (Appendix H),
// f_n = n! C((m+n)/2 - 1, n/2), S_{A,B}(i, j) = [x_{A_i} = x_{B_j}] (so Per is
// the product of c! over the values whose multiplicities c in A and B agree,
// and 0 if any disagree). W_T is W on the rows/columns x_T. (The pseudocode's
// e' uses s; the theorem's B ranges over [k] \ a. Both are read with s', which
// the brute-force marginal of Eq. marginal_definition confirms.)
//
// Evaluation order. The same sum, regrouped by rho = [k] \ A: Per(S_{A,B})
// vanishes unless A and B hold the same multiset alpha of modes, and is then
// prod_v alpha_v!; rho_A and rho_B then hold equal multisets too, so their
// sub-Hafnians agree, and for fixed A the sum over s runs over s in rho_A:
//   q_n = sum_rho w(rho) sum_{ja, jb} F(k, k - |rho|, ja, jb) / f_n G(rho, ja) conj(G(rho, jb)),
//   G(rho, j) = sum_{sigma in rho, |sigma| = j} Haf(W_sigma) Haf(W_{rho \ sigma}),
//   w(rho) = prod_v alpha_v! C(m_v, alpha_v)
// (alpha_v = m_v - |rho cap positions of v|, m_v the multiplicity of mode v in
// the prefix; C(m_v, alpha_v) counts the sets B with A's multiset; w = 1
// without repeated modes, the Proposition). A perfect matching of sigma with
// one of rho \ sigma is a perfect matching of rho with j / 2 of its pairs
// marked, so G(rho, j) = C(|rho| / 2, j / 2) Haf(W_rho), and the sum over the
// subsets sigma (3^k products in all) is gone:
//   q_n = sum_rho w(rho) c_k(|rho|) |Haf(W_rho)|^2,
//   c_k(s) = sum_{ja, jb} F(k, k - s, ja, jb) / f_n C(s/2, ja/2) C(s/2, jb/2)
// over the (ja, jb) inside the theorem's ranges (F is 0 outside them).
//
// The sub-Hafnians come from each other by expanding along one row,
//   Haf(B_T) = sum_{i in T, i != p} B(x_p, x_i) Haf(B_{T \ {p, i}}),
// so a prefix's table costs at most k - 1 complex products an entry. Tables
// hold the even sets only, at index T >> 1 (the lowest bit follows from the
// parity), and Haf(B_T) rather than Haf(W_T): c_k absorbs tanh(r)^{-s} (for a
// tiny r both with g B, see b_unit).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "gbs_api_internal.h"

namespace gbs {
namespace {

constexpr int kMaxK = 20;  // prefix length limit (position masks in an int; tables of 2^(k-1) sets)
constexpr int kMargThreads = 256;
constexpr int kCoefs = kMaxK / 2 + 1;  // c_k(0), c_k(2), .. per prefix length

// C(p, i) for p, i <= kMaxK (Pascal's rule, at compile time), in global
// memory; blocks copy it (coalesced) into shared memory, where lanes index it
// freely.
struct BinomTable {
  int v[kMaxK + 1][kMaxK + 1];
};
constexpr BinomTable make_binom_table() {
  BinomTable t{};
  for (int p = 0; p <= kMaxK; ++p)
    for (int i = 0; i <= kMaxK; ++i) t.v[p][i] = i == 0 ? 1 : p == 0 ? 0 : t.v[p - 1][i - 1] + t.v[p - 1][i];
  return t;
}
__device__ const BinomTable c_binom = make_binom_table();
static_assert(make_binom_table().v[20][10] == 184756, "Pascal table");

// Rows p <= rows of the table (a prefix of length k indexes p < k).
__device__ __forceinline__ void load_binom(int (*binom)[kMaxK + 1], int rows) {
  for (int q = threadIdx.x; q < (rows + 1) * (kMaxK + 1); q += blockDim.x)
    binom[q / (kMaxK + 1)][q % (kMaxK + 1)] = c_binom.v[q / (kMaxK + 1)][q % (kMaxK + 1)];
}

// q_n does not depend on t = tanh r > 0, but |Haf(B_T)|^2 ~ t^{|T|} leaves the
// range of a double from t ~ 1e-16 on at 20 photons. Below 2^-16 the sums
// therefore read g B, a copy made for the call with a power of two g (exact)
// that puts g t into [1, 2); above, g = 1 and they read B itself. (Multiplying
// by g wherever a set's Hafnian is formed cost ordinary calls up to 10 %.)
double b_unit(double t) { return t < 0x1p-16 ? ldexp(1.0, std::min(-ilogb(t), 1022)) : 1.0; }
__global__ void scale_kernel(const double* __restrict__ B, double* __restrict__ gB, int64_t count, double g) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
    gB[i] = g * B[i];
}
// What the sums read: k's B, or its copy at `copy` (b_copy_bytes of scratch).
size_t b_copy_bytes(const gbs_kernel* k) { return b_unit(k->t_uniform) == 1.0 ? 0 : 16 * (size_t)k->m * k->m; }
const double* scaled_B(const gbs_kernel* k, void* copy, cudaStream_t st) {
  const double g = b_unit(k->t_uniform);
  if (g == 1.0) return k->B;
  const int64_t count = 2 * (int64_t)k->m * k->m;
  scale_kernel<<<(int)std::min<int64_t>(8192, (count + 255) / 256), 256, 0, st>>>(k->B, (double*)copy, count, g);
  return (const double*)copy;
}

// (g t)^{-s} for s = 0..kMaxK: |Haf(W_T)|^2 = (g t)^{-|T|} |Haf(g B_T)|^2.
// Computed once per call on the host.
struct SizeScale {
  double s[kMaxK + 1];
};

SizeScale size_scale(double t) {
  const double gt = b_unit(t) * t;
  SizeScale sc;
  for (int i = 0; i <= kMaxK; ++i) {
    const double h = pow(gt, -0.5 * i);
    sc.s[i] = h * h;
  }
  return sc;
}

// The ranges of Theorem 1: ja, jb (the even sizes of s and s') at least
// max(0, 2k - n), and mu = |A| in [max(0, 3k - ja - jb - n), k - max(ja, jb)].
// F vanishes outside them, so no term there is formed.
__host__ __device__ __forceinline__ bool theorem_range(int k, int n, int mu, int ja, int jb) {
  const int lo = 2 * k - n > 0 ? 2 * k - n : 0;
  const int hi = ja > jb ? ja : jb;
  return ja >= lo && jb >= lo && mu >= (3 * k - ja - jb - n > 0 ? 3 * k - ja - jb - n : 0) && mu <= k - hi;
}

// Bit s set if c_k(s) has a term in range.
unsigned rho_sizes(int k, int n) {
  unsigned sizes = 0;
  for (int c = 0; c <= k; c += 2)
    for (int ja = 0; ja <= c; ja += 2)
      for (int jb = 0; jb <= c; jb += 2)
        if (theorem_range(k, n, k - c, ja, jb)) sizes |= 1u << c;
  return sizes;
}

// c_k(s) (g t)^{-s}, s = 0, 2, .., k, of prefix length k = k0 + blockIdx.x at
// out + k * kCoefs. The log-gammas take few distinct arguments (by mu, by
// ja + jb and by mu + ja + jb), one thread each; a thread per term evaluated
// seven in a row, 28 us for a launch, against 10 us now.
__global__ void __launch_bounds__(kMargThreads) coef_kernel(int k0, int n, int m, SizeScale scale,
                                                            double* __restrict__ out) {
  constexpr int kA = kMaxK + 1, kC = 3 * kMaxK + 1, kR = kMaxK / 2 + 1;
  __shared__ double LA[kA], LB[kA], LC[kC], L0[5];
  __shared__ double term[kR * kR * kR];
  __shared__ int binom[kMaxK + 1][kMaxK + 1];
  const int k = k0 + (int)blockIdx.x;
  load_binom(binom, kMaxK);
  const double hm = 0.5 * m;
  for (int q = threadIdx.x; q < 2 * kA + kC + 5; q += blockDim.x) {
    if (q < kA) {
      LA[q] = lgamma(0.5 * (n - k + q + m));  // q = mu
    } else if (q < 2 * kA) {
      const int s = q - kA;  // (ja + jb) / 2
      LB[s] = lgamma(k - s + hm);
    } else if (q < 2 * kA + kC) {
      const int e = q - 2 * kA;  // mu + ja + jb
      LC[e] = lgamma(0.5 * (n - k + e) - k + 1.0);
    } else {
      const int i = q - 2 * kA - kC;
      const double a = i == 0 ? n - k + 1.0 : i == 1 ? n + 1.0 : i == 2 ? 0.5 * (m + n) : i == 3 ? 0.5 * n + 1.0 : hm;
      L0[i] = lgamma(a);
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < kR * kR * kR; q += blockDim.x) {
    const int r = q / (kR * kR), a = (q / kR) % kR, b = q % kR, c = 2 * r, mu = k - c;
    double v = 0.0;
    if (c <= k && a <= r && b <= r && theorem_range(k, n, mu, 2 * a, 2 * b))
      v = exp(L0[0] + (LA[mu] - LB[a + b] - LC[mu + 2 * (a + b)]) - L0[1] - (L0[2] - L0[3] - L0[4])) *
          ((double)binom[r][a] * (double)binom[r][b]);
    term[q] = v;
  }
  __syncthreads();
  if (threadIdx.x < kR && 2 * threadIdx.x <= k) {
    const int r = threadIdx.x;
    double s = 0.0;
    for (int a = 0; a <= r; ++a)
      for (int b = 0; b <= r; ++b) s += term[(r * kR + a) * kR + b];
    out[(int64_t)k * kCoefs + r] = s * scale.s[2 * r];
  }
}

// The subsets of `bits` positions with the sizes t[i] (C(bits, t[i]) each,
// numbered from start[i]), largest sizes first.
struct SubsetClasses {
  int bits = 0, ncls = 0;
  int t[kMaxK + 1];
  int64_t start[kMaxK + 2];
  __host__ __device__ int64_t total() const { return start[ncls]; }
};

// The subsets of `bits` positions of size s - shift for the sizes s marked in
// `sizes` (bit s).
SubsetClasses subset_classes(int bits, unsigned sizes, int shift) {
  SubsetClasses sc;
  sc.bits = bits;
  sc.start[0] = 0;
  for (int s = kMaxK; s >= 0; --s) {
    const int t = s - shift;
    if (!(sizes >> s & 1u) || t < 0 || t > bits) continue;
    int64_t cnt = 1;
    for (int i = 1; i <= t; ++i) cnt = cnt * (bits - t + i) / i;
    sc.t[sc.ncls] = t;
    sc.start[sc.ncls + 1] = sc.start[sc.ncls] + cnt;
    ++sc.ncls;
  }
  return sc;
}

// The t-subset of `bits` positions of colex rank `rank` (rank = sum_i C(p_i, i)
// over the positions p_1 < .. < p_t).
__device__ __forceinline__ int unrank(int bits, int t, int rank, const int (*binom)[kMaxK + 1]) {
  int mask = 0;
  for (int i = t, p = bits - 1; i >= 1; --i) {
    while (binom[p][i] > rank) --p;
    mask |= 1 << p;
    rank -= binom[p][i];
    --p;
  }
  return mask;
}
// Entry r of the classes: its size class, then its rank.
__device__ __forceinline__ int subset_of(const SubsetClasses& sc, int64_t r, const int (*binom)[kMaxK + 1]) {
  int cls = 0;
  while (r >= sc.start[cls + 1]) ++cls;
  return unrank(sc.bits, sc.t[cls], (int)(r - sc.start[cls]), binom);
}

__device__ __forceinline__ void cfma_acc(double2& acc, double2 a, double2 b) {
  acc.x = fma(a.x, b.x, acc.x);
  acc.x = fma(-a.y, b.y, acc.x);
  acc.y = fma(a.x, b.y, acc.y);
  acc.y = fma(a.y, b.x, acc.y);
}

// sum_{i in T} row(i) Haf(T \ i), T odd, from a table of even sets. The terms
// are added in increasing position order.
template <class Row>
__device__ __forceinline__ double2 expand(const double2* H, int T, const Row& row) {
  double2 acc = make_double2(0.0, 0.0);
  for (int rest = T; rest; rest &= rest - 1) {
    const int i = __ffs(rest) - 1;
    cfma_acc(acc, row(i), H[(T ^ (1 << i)) >> 1]);
  }
  return acc;
}

// The modes that a prefix holds more than once: position masks and counts
// (a mode held once has weight 1 either way).
struct Repeats {
  int n, mask[kMaxK], mult[kMaxK], mode[kMaxK];
};
__device__ void find_repeats(Repeats& R, const int* x, int k) {
  int r = 0;
  unsigned seen = 0;
  for (int i = 0; i < k; ++i) {
    if (seen >> i & 1u) continue;
    int mask = 1 << i;
    for (int j = i + 1; j < k; ++j)
      if (x[j] == x[i]) mask |= 1 << j;
    seen |= (unsigned)mask;
    if (mask != (1 << i)) {
      R.mask[r] = mask;
      R.mult[r] = __popc(mask);
      R.mode[r] = x[i];
      ++r;
    }
  }
  R.n = r;
}
// w(rho), at most 20! and exact; with `extra` = r >= 0 mode r of the list
// counts one copy more, outside rho's positions but in rho (C(m+1, alpha)).
__device__ __forceinline__ double rho_weight(const Repeats& R, int rho, const int (*binom)[kMaxK + 1], int extra = -1) {
  int64_t w = 1;
  for (int v = 0; v < R.n; ++v) {
    const int mv = R.mult[v], al = mv - __popc(rho & R.mask[v]);
    for (int i = 2; i <= al; ++i) w *= i;
    w *= binom[mv + (v == extra ? 1 : 0)][al];
  }
  return (double)w;
}

// A block's sum in a fixed tree.
__device__ __forceinline__ double block_sum(double v, double* red) {
  red[threadIdx.x] = v;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  return red[0];
}

// Prefixes of up to kMargSmem photons: one block each, the table in shared
// memory, built size by size (each set along its lowest position's row) with
// the sum taken as the sets are formed. The latency of a few layers bounds it.
// A call for 256 prefixes of 9 photons (n = 16) takes 82 us, launches and the
// result's copy included; with index lists built on the host, batched Hafnians
// and the sum over subsets sigma it took 3.44 ms.
constexpr int kMargSmem = 12;
__global__ void __launch_bounds__(kMargThreads) marginal_small_kernel(int k, const double2* __restrict__ B, int m,
                                                                      const int* x, unsigned sizes,
                                                                      const double* coef, double* q) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int binom[kMaxK + 1][kMaxK + 1];
  __shared__ double2 Bx[kMargSmem * kMargSmem];
  __shared__ int xs[kMaxK];
  __shared__ Repeats R;
  __shared__ double red[kMargThreads];
  double2* H = reinterpret_cast<double2*>(smem);
  load_binom(binom, kMaxK);
  dependency_wait();
  if (threadIdx.x < k) xs[threadIdx.x] = x[(int64_t)blockIdx.x * k + threadIdx.x];
  if (threadIdx.x == 0) H[0] = make_double2(1.0, 0.0);
  __syncthreads();
  if (threadIdx.x == 0) find_repeats(R, xs, k);
  for (int e = threadIdx.x; e < k * k; e += blockDim.x) Bx[e] = __ldg(B + (int64_t)xs[e / k] * m + xs[e % k]);
  __syncthreads();
  double acc = 0.0;
  if (threadIdx.x == 0 && (sizes & 1u)) acc = coef[0] * (R.n ? rho_weight(R, 0, binom) : 1.0);
  const int top = 31 - __clz((int)(sizes | 1u));
  for (int s = 2; s <= top; s += 2) {
    const double c = (sizes >> s & 1u) ? coef[s / 2] : 0.0;
    for (int r = threadIdx.x; r < binom[k][s]; r += blockDim.x) {
      const int T = unrank(k, s, r, binom), p = __ffs(T) - 1;
      const double2* row = Bx + p * k;
      const double2 h = expand(H, T & (T - 1), [&](int i) { return row[i]; });
      H[T >> 1] = h;
      if (c != 0.0) acc = fma(c * (R.n ? rho_weight(R, T, binom) : 1.0), h.x * h.x + h.y * h.y, acc);
    }
    __syncthreads();
  }
  const double sum = block_sum(acc, red);
  if (threadIdx.x == 0) q[blockIdx.x] = sum;
}

// Longer prefixes: the tables in device memory, one launch per size.
__global__ void __launch_bounds__(kMargThreads) marginal_layer_kernel(int k, int s, const double2* __restrict__ B, int m,
                                                                      const int* __restrict__ x, int batch,
                                                                      double2* __restrict__ H) {
  __shared__ int binom[kMaxK + 1][kMaxK + 1];
  load_binom(binom, kMaxK);
  __syncthreads();
  const int cnt = binom[k][s];
  const int64_t all = (int64_t)batch * cnt;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < all; q += (int64_t)gridDim.x * blockDim.x) {
    const int b = (int)(q / cnt), T = unrank(k, s, (int)(q - (int64_t)b * cnt), binom);
    const int* xs = x + (int64_t)b * k;
    double2* Hb = H + ((int64_t)b << (k - 1));
    if (s == 0) {
      Hb[0] = make_double2(1.0, 0.0);
      continue;
    }
    const double2* row = B + (int64_t)xs[__ffs(T) - 1] * m;
    Hb[T >> 1] = expand(Hb, T & (T - 1), [&](int i) { return __ldg(row + xs[i]); });
  }
}

// q of prefix blockIdx.x from its sub-Hafnians: entry j of the classes has its
// set's Hafnian at H[b * stride + T >> 1], or (list) at H[b * stride + j].
__global__ void __launch_bounds__(kMargThreads) marginal_sum_kernel(int k, SubsetClasses rho, bool list,
                                                                    const int* __restrict__ x,
                                                                    const double2* __restrict__ H, int64_t stride,
                                                                    const double* __restrict__ coef,
                                                                    double* __restrict__ q) {
  __shared__ int binom[kMaxK + 1][kMaxK + 1];
  __shared__ Repeats R;
  __shared__ double red[kMargThreads];
  load_binom(binom, kMaxK);
  if (threadIdx.x == 0) find_repeats(R, x + (int64_t)blockIdx.x * k, k);
  __syncthreads();
  double acc = 0.0;
  for (int64_t j = threadIdx.x; j < rho.total(); j += blockDim.x) {
    const int T = subset_of(rho, j, binom);
    const double2 h = H[blockIdx.x * stride + (list ? j : T >> 1)];
    acc = fma(coef[__popc(T) / 2] * (R.n ? rho_weight(R, T, binom) : 1.0), h.x * h.x + h.y * h.y, acc);
  }
  const double sum = block_sum(acc, red);
  if (threadIdx.x == 0) q[blockIdx.x] = sum;
}

// ---- the chain sampler ----------------------------------------------------
//
// Exponential-space variant (Appendix D): each sample keeps the sub-Hafnians
// of its prefix. A set rho that holds the new photon (mode l) is T plus it, T
// odd, and Haf(B_rho) = sum_{i in T} B(l, x_i) h_i, h_i = Haf(B_{T \ i}) from
// the prefix. For a mode l outside the prefix w(rho) does not depend on l, so
// its sum over those sets is a Hermitian form in the row b_i = B(l, x_i):
//   sum_T w(T) c_k(|T| + 1) |sum_i b_i h_i|^2 = b* M b,
//   M_ij = sum_{T holds i, j} w(T) c_k(|T| + 1) conj(h_i) h_j,
// and M serves every candidate of the sample: k^2 / 2 products a candidate
// instead of up to k 2^(k-2). A mode in the prefix has one copy more, and with
// it a larger weight on the sets that do not hold all its positions: what it
// has more there (every term positive) is summed apart, for at most k - 1
// modes. On the last step, with one set, all candidates are summed one by one.
// The sets without
// the new photon count 1 + (multiplicity of l in the prefix) times:
// (a+1)! C(m+1, a+1) = (m+1) a! C(m, a). 64 samples of 16 photons over 256
// modes: 9.56 ms (every candidate's table and sums over subsets) -> 0.80 ms.
struct ChainStep {
  int k, n, m, kp;           // kp = k - 1 photons in the prefix
  bool direct;               // every candidate one by one: no M
  SubsetClasses rho;         // sets of the prefix that count (even)
  SubsetClasses odd;         // sets T of the prefix with c_k(|T| + 1) in range
  SubsetClasses pair, diag;  // T without two (one) of its positions, over the other kp - 2 (kp - 1)
  SubsetClasses miss;        // sets T that do not hold one given position, over the other kp - 1
  SubsetClasses grow;        // odd sets whose union with the new photon a later step reads
  int n_pair, c_pair, c_own, c_rho;  // position pairs i <= j; warps of each, of a prefix mode, of the rho sum
  int tasks;                 // warps per sample
};
constexpr int kPairChunk = 256, kOwnChunk = 64, kRhoChunk = 512;  // sets per warp

// Inserts a zero bit at position i.
__device__ __forceinline__ int open_bit(int v, int i) { return ((v >> i) << (i + 1)) | (v & ((1 << i) - 1)); }

__device__ __forceinline__ double warp_sum(double v) {
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// One warp per task of sample blockIdx.y: a chunk of M_ij, of what one prefix
// mode has more (that of position t, by its first position; 0 for others) or
// of the sum over rho. part[sample * tasks + task]. A mode held once (the
// common case) has weight 2 instead of 1 on the sets without its position, so
// half the sets are enough for it; a repeated one goes through all of them.
__global__ void __launch_bounds__(kMargThreads) chain_gram_kernel(ChainStep S, const double2* cache,
                                                                  int64_t cstride, const double2* __restrict__ B,
                                                                  const int* x, const double* coefs, double2* part) {
  __shared__ int binom[kMaxK + 1][kMaxK + 1];
  __shared__ Repeats R;
  __shared__ int xs[kMaxK];
  __shared__ double coef[kCoefs];
  const int smp = blockIdx.y, lane = threadIdx.x & 31;
  load_binom(binom, kMaxK);
  dependency_wait();
  if (threadIdx.x < S.kp) xs[threadIdx.x] = x[(int64_t)smp * kMaxK + threadIdx.x];
  if (threadIdx.x < kCoefs) coef[threadIdx.x] = 2 * threadIdx.x <= S.k ? coefs[(int64_t)S.k * kCoefs + threadIdx.x] : 0.0;
  __syncthreads();
  if (threadIdx.x == 0) find_repeats(R, xs, S.kp);
  __syncthreads();
  const double2* H = cache + (int64_t)smp * cstride;
  auto weight = [&](int T, int size, int extra = -1) {
    return coef[size / 2] * (R.n ? rho_weight(R, T, binom, extra) : 1.0);
  };
  const int task = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (task >= S.tasks) return;
  int t = task;
  double re = 0.0, im = 0.0;
  if (t < S.n_pair * S.c_pair) {
    const int pr = t / S.c_pair, c0 = (t - pr * S.c_pair) * kPairChunk;
    int j = 0;
    while ((j + 1) * (j + 2) / 2 <= pr) ++j;
    const int i = pr - j * (j + 1) / 2;  // i <= j
    if (i == j) {
      const int end = (int)min(S.diag.total(), (int64_t)c0 + kPairChunk);
      for (int r = c0 + lane; r < end; r += 32) {
        const int U = open_bit(subset_of(S.diag, r, binom), i), T = U | (1 << i);
        const double2 h = H[U >> 1];
        re = fma(weight(T, __popc(T) + 1), h.x * h.x + h.y * h.y, re);
      }
    } else {
      const int end = (int)min(S.pair.total(), (int64_t)c0 + kPairChunk);
      for (int r = c0 + lane; r < end; r += 32) {
        const int U = open_bit(open_bit(subset_of(S.pair, r, binom), i), j), T = U | (1 << i) | (1 << j);
        const double2 hi = H[(U | (1 << j)) >> 1], hj = H[(U | (1 << i)) >> 1];
        const double w = weight(T, __popc(T) + 1);
        re = fma(w, fma(hi.x, hj.x, hi.y * hj.y), re);
        im = fma(w, fma(hi.x, hj.y, -hi.y * hj.x), im);
      }
    }
  } else if ((t -= S.n_pair * S.c_pair) < S.kp * S.c_own) {
    const int p = t / S.c_own, c0 = (t - p * S.c_own) * kOwnChunk, v = xs[p];
    int first = p;
    for (int i = p - 1; i >= 0; --i)
      if (xs[i] == v) first = i;
    if (first == p) {
      int extra = -1;
      for (int i = 0; i < R.n; ++i)
        if (R.mode[i] == v) extra = i;
      const double2* row = B + (int64_t)v * S.m;
      const int end = (int)min(extra < 0 ? S.miss.total() : S.odd.total(), (int64_t)c0 + kOwnChunk);
      for (int r = c0 + lane; r < end; r += 32) {
        const int T = extra < 0 ? open_bit(subset_of(S.miss, r, binom), p) : subset_of(S.odd, r, binom);
        double w = weight(T, __popc(T) + 1);
        if (extra >= 0) {  // (m + 1) / (m + 1 - alpha) times as much, alpha of m copies outside T
          const int mv = R.mult[extra], al = mv - __popc(T & R.mask[extra]);
          if (al == 0) continue;
          w = weight(T, __popc(T) + 1, extra) - w;
        }
        const double2 h = expand(H, T, [&](int i) { return __ldg(row + xs[i]); });
        re = fma(w, h.x * h.x + h.y * h.y, re);
      }
    }
  } else {
    t -= S.kp * S.c_own;
    const int c0 = t * kRhoChunk, end = (int)min(S.rho.total(), (int64_t)c0 + kRhoChunk);
    for (int r = c0 + lane; r < end; r += 32) {
      const int T = subset_of(S.rho, r, binom);
      const double2 h = H[T >> 1];
      re = fma(weight(T, __popc(T)), h.x * h.x + h.y * h.y, re);
    }
  }
  re = warp_sum(re);
  im = warp_sum(im);
  if (lane == 0) part[(int64_t)smp * S.tasks + task] = make_double2(re, im);
}

// The candidates' weights q[sample * m + l], a thread each (sample
// blockIdx.y); the chunks of the gram kernel are added in their order.
constexpr int kWeightThreads = 128;
__global__ void __launch_bounds__(kWeightThreads) chain_weight_kernel(ChainStep S, const double2* cache,
                                                                      int64_t cstride, const double2* __restrict__ B,
                                                                      const int* x, const double* coefs,
                                                                      const double2* part, double* q) {
  __shared__ double2 M[kMaxK * (kMaxK + 1) / 2], b[kMaxK][kWeightThreads];
  __shared__ double own[kMaxK], s_rho;
  __shared__ int xs[kMaxK], binom[kMaxK + 1][kMaxK + 1];
  __shared__ Repeats R;
  __shared__ double coef[kCoefs];
  const int smp = blockIdx.y, l = blockIdx.x * kWeightThreads + threadIdx.x;
  const double2* ps = part + (int64_t)smp * S.tasks;
  if (S.direct) load_binom(binom, kMaxK);
  dependency_wait();
  if (S.direct) {
    if (threadIdx.x < kCoefs) coef[threadIdx.x] = 2 * threadIdx.x <= S.k ? coefs[(int64_t)S.k * kCoefs + threadIdx.x] : 0.0;
  }
  if (threadIdx.x < S.kp) xs[threadIdx.x] = x[(int64_t)smp * kMaxK + threadIdx.x];
  const int n_own = S.c_own > 0 ? S.kp : 0;
  for (int e = threadIdx.x; e < S.n_pair + n_own + 1; e += blockDim.x) {
    const bool pr = e < S.n_pair, ow = !pr && e < S.n_pair + n_own;
    const int cnt = pr ? S.c_pair : ow ? S.c_own : S.c_rho;
    const double2* p = ps + (pr ? e * S.c_pair : S.n_pair * S.c_pair + (ow ? (e - S.n_pair) * S.c_own : S.kp * S.c_own));
    double2 s = make_double2(0.0, 0.0);
    for (int c = 0; c < cnt; ++c) {
      s.x += p[c].x;
      s.y += p[c].y;
    }
    if (pr) M[e] = s;
    else if (ow) own[e - S.n_pair] = s.x;
    else s_rho = s.x;
  }
  __syncthreads();
  if (S.direct && threadIdx.x == 0) find_repeats(R, xs, S.kp);
  if (l < S.m)
    for (int i = 0; i < S.kp; ++i) b[i][threadIdx.x] = __ldg(B + (int64_t)l * S.m + xs[i]);
  __syncthreads();
  if (l >= S.m) return;
  int mult = 0, first = -1;
  for (int i = S.kp - 1; i >= 0; --i)
    if (xs[i] == l) {
      ++mult;
      first = i;
    }
  double s = 0.0;
  if (S.direct) {
    int extra = -1;
    for (int i = 0; i < R.n; ++i)
      if (R.mode[i] == l) extra = i;
    const double2* H = cache + (int64_t)smp * cstride;
    for (int r = 0; r < (int)S.odd.total(); ++r) {
      const int T = subset_of(S.odd, r, binom);
      const double2 h = expand(H, T, [&](int i) { return b[i][threadIdx.x]; });
      double w = coef[(__popc(T) + 1) / 2] * (R.n ? rho_weight(R, T, binom, extra) : 1.0);
      if (mult == 1 && !(T >> first & 1)) w *= 2.0;
      s = fma(w, h.x * h.x + h.y * h.y, s);
    }
  } else {
    if (mult > 0) s = own[first];
    for (int i = 0; i < S.kp; ++i) {
      const double2 bi = b[i][threadIdx.x];
      double2 y = make_double2(0.0, 0.0);  // sum_{j > i} M_ij b_j
      for (int j = i + 1; j < S.kp; ++j) cfma_acc(y, M[j * (j + 1) / 2 + i], b[j][threadIdx.x]);
      s = fma(M[i * (i + 1) / 2 + i].x, bi.x * bi.x + bi.y * bi.y, s);
      s = fma(2.0, bi.x * y.x + bi.y * y.y, s);
    }
  }
  q[(int64_t)smp * S.m + l] = fmax(fma(1.0 + mult, s_rho, s), 0.0);
}

// Every cache starts as Haf of the empty matrix, 1.
__global__ void chain_init_kernel(double2* __restrict__ cache, int64_t cstride, int samples) {
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < samples; s += gridDim.x * blockDim.x)
    cache[s * cstride] = make_double2(1.0, 0.0);
}

// Step k's draw for sample blockIdx.y, then (k < n) its cache update; every
// block of the sample draws (the same inputs give the same mode) and updates
// its share of the cache. The draw, by warp 0: the running sums of the weights
// in mode order (each lane a contiguous run of modes, the runs joined by a
// fixed warp scan), and x_k = the first l of positive weight whose running sum
// exceeds u_k times the total (m - 1 if there is none); block 0 writes it. The
// update: the sets of x_k with the odd T' that later steps read.
//   u: n uniforms per sample; x: kMaxK sampled modes per sample.
constexpr int kPickModes = 2048;
__global__ void __launch_bounds__(kMargThreads) chain_pick_kernel(ChainStep S, const double* q, const double* u, int* x,
                                                                  double2* cache, int64_t cstride,
                                                                  const double2* __restrict__ B) {
  __shared__ int s_pick;
  __shared__ int binom[kMaxK + 1][kMaxK + 1], xs[kMaxK];
  __shared__ double s_q[kPickModes];  // the weights, where they fit
  const int smp = blockIdx.y, m = S.m;
  if (S.k < S.n) load_binom(binom, kMaxK);
  dependency_wait();
  if (threadIdx.x < S.kp) xs[threadIdx.x] = x[(int64_t)smp * kMaxK + threadIdx.x];
  const bool fits = m <= kPickModes;
  if (fits) {
    for (int l = threadIdx.x; l < m; l += blockDim.x) s_q[l] = q[(int64_t)smp * m + l];
    __syncthreads();
  }
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    const double* qs = fits ? s_q : q + (int64_t)smp * m;
    const int per = (m + 31) / 32, lo = min(m, lane * per), hi = min(m, lo + per);
    double part = 0.0;
    for (int l = lo; l < hi; ++l) part += qs[l];
    double inc = part;  // inclusive scan over the lanes, fixed order
    for (int off = 1; off < 32; off <<= 1) {
      const double v = __shfl_up_sync(0xffffffffu, inc, off);
      if (lane >= off) inc += v;
    }
    const double tot = __shfl_sync(0xffffffffu, inc, 31);
    double run = __shfl_up_sync(0xffffffffu, inc, 1);
    if (lane == 0) run = 0.0;
    const double target = u[(int64_t)smp * S.n + S.k - 1] * tot;
    int found = m;
    for (int l = lo; l < hi; ++l) {
      const double w = qs[l];
      run += w;
      if (w > 0.0 && run > target) {
        found = l;
        break;
      }
    }
    const unsigned ball = __ballot_sync(0xffffffffu, found < m);
    const int first = __shfl_sync(0xffffffffu, found, ball ? __ffs(ball) - 1 : 0);
    if (lane == 0) s_pick = ball ? first : m - 1;
  }
  __syncthreads();
  const int pick = s_pick;
  if (blockIdx.x == 0 && threadIdx.x == 0) x[(int64_t)smp * kMaxK + S.kp] = pick;
  if (S.k == S.n) return;
  double2* c = cache + (int64_t)smp * cstride;
  const double2* row = B + (int64_t)pick * m;
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < (int)S.grow.total(); r += gridDim.x * blockDim.x) {
    const int T = subset_of(S.grow, r, binom);
    c[(T | (1 << S.kp)) >> 1] = expand(c, T, [&](int i) { return __ldg(row + xs[i]); });
  }
}

int64_t choose(int a, int b) {
  if (b < 0 || b > a) return 0;
  int64_t v = 1;
  for (int i = 1; i <= b; ++i) v = v * (a - b + i) / i;
  return v;
}

// Step k of n over m modes; `later` (bit s) marks the sizes of new sets that
// steps after k read.
ChainStep chain_step(int k, int n, int m, unsigned later) {
  ChainStep S;
  S.k = k;
  S.n = n;
  S.m = m;
  S.kp = k - 1;
  const unsigned sizes = rho_sizes(k, n);
  S.rho = subset_classes(S.kp, sizes, 0);
  S.odd = subset_classes(S.kp, sizes, 1);
  S.pair = subset_classes(std::max(S.kp - 2, 0), S.kp >= 2 ? sizes : 0, 3);
  S.diag = subset_classes(std::max(S.kp - 1, 0), S.kp >= 1 ? sizes : 0, 2);
  S.miss = S.kp >= 1 ? subset_classes(S.kp - 1, sizes, 1) : SubsetClasses();
  S.grow = subset_classes(S.kp, later, 1);
  // a candidate costs kp products per set one by one and kp / 2 per position by
  // the form (at k = n there is one set; at k = n - 1 of 16, 14 sets one by one
  // took 87 us for 64 samples, the form 40 with its sums)
  S.direct = 2 * S.odd.total() <= S.kp;
  auto chunks = [](int64_t total, int per) { return (int)std::max<int64_t>(1, (total + per - 1) / per); };
  S.n_pair = S.direct ? 0 : S.kp * (S.kp + 1) / 2;
  S.c_pair = S.direct ? 0 : chunks(std::max(S.pair.total(), S.diag.total()), kPairChunk);
  S.c_own = S.direct ? 0 : chunks(S.odd.total(), kOwnChunk);
  S.c_rho = chunks(S.rho.total(), kRhoChunk);
  S.tasks = S.n_pair * S.c_pair + S.kp * S.c_own + S.c_rho;
  return S;
}

}  // namespace
}  // namespace gbs

using namespace gbs;

extern "C" int gbs_marginal_batch(const gbs_kernel* k, const int* x, int kk, int batch, int n, void* stream,
                                  double* q_out) {
  clear_error();
  if (!k || (batch > 0 && (!q_out || (kk > 0 && !x)))) return fail(GBS_EINVAL, "null argument");
  if (batch < 0) return fail(GBS_EINVAL, "batch = %d is negative", batch);
  if (batch == 0) return GBS_OK;
  if (n < 0 || n > GBS_MAX_N || (n & 1)) return fail(GBS_ERANGE, "n = %d must be even and <= %d", n, GBS_MAX_N);
  if (kk < 0 || kk > n || kk > kMaxK) return fail(GBS_ERANGE, "prefix length %d outside [0, min(n, %d)]", kk, kMaxK);
  if (!k->r_uniform) return fail(GBS_EINVAL, "marginals need identical squeezing on every mode");
  if (!(k->t_uniform > 0.0)) return fail(GBS_EINVAL, "marginals need r > 0");
  cudaStream_t st = (cudaStream_t)stream;
  // prefixes on the host (small), to check them
  std::vector<int> hx((size_t)batch * std::max(kk, 1));
  if (kk > 0) {
    const cudaError_t e0 = cudaMemcpy(hx.data(), x, sizeof(int) * batch * kk, cudaMemcpyDefault);
    if (e0 != cudaSuccess) return cuda_fail(e0, "prefix copy");
  }
  for (size_t i = 0; i < (size_t)batch * kk; ++i)
    if (hx[i] < 0 || hx[i] >= k->m) return fail(GBS_ERANGE, "mode index %d outside [0, %d)", hx[i], k->m);
  const unsigned sizes = rho_sizes(kk, n);
  const SubsetClasses rho = subset_classes(kk, sizes, 0);
  // Long prefixes near n need few, large sets: those come cheaper one by one
  // from the batched Hafnians (at k = n = 20 one set of 90 thousand complex
  // products, against 5 million for its table).
  double table = 0.0, single = 0.0;
  int top = 0;
  for (int s = 2; s <= kk; s += 2) {
    double macs;
    int even, odd;
    match_sizes(s, &even, &odd, &macs);
    if (sizes >> s & 1u) {
      single += (double)choose(kk, s) * macs;
      top = s;
    }
  }
  for (int s = 2; s <= top; s += 2) table += (double)choose(kk, s) * (s - 1);
  const bool list = kk > kMargSmem && single < table;
  const bool small = !list && kk <= kMargSmem;
  const int64_t stride = list ? rho.total() : small ? 0 : (int64_t)1 << (kk - 1);
  // tables of at most 2 GB at once
  const int64_t group = small ? batch : std::max<int64_t>(1, std::min<int64_t>(batch, ((int64_t)1 << 27) / stride));
  auto al = [](size_t v) { return (v + 255) & ~(size_t)255; };
  const size_t H_b = al(16 * (size_t)(small ? 0 : group * stride)), c_b = al(8 * (size_t)(kMaxK + 1) * kCoefs);
  const size_t x_b = al(4 * hx.size()), q_b = al(8 * (size_t)batch), B_b = al(b_copy_bytes(k));
  void* tmp = nullptr;
  cudaError_t e = scratch_alloc(&tmp, H_b + c_b + x_b + q_b + B_b, st);
  if (e != cudaSuccess) return fail(GBS_ENOMEM, "marginal scratch: %s", cudaGetErrorString(e));
  unsigned char* t = (unsigned char*)tmp;
  double2* d_H = (double2*)t;
  double* d_c = (double*)(t + H_b);
  int* d_x = (int*)(t + H_b + c_b);
  double* d_q = (double*)(t + H_b + c_b + x_b);
  const bool q_dev = is_device_ptr(q_out);
  const double2* B = (const double2*)scaled_B(k, t + H_b + c_b + x_b + q_b, st);
  const double* coef = d_c + (size_t)kk * kCoefs;
  int ret = GBS_OK;
  do {
    if (kk > 0 && (e = cudaMemcpyAsync(d_x, hx.data(), 4 * hx.size(), cudaMemcpyHostToDevice, st)) != cudaSuccess) {
      ret = cuda_fail(e, "marginal upload");
      break;
    }
    coef_kernel<<<1, kMargThreads, 0, st>>>(kk, n, k->m, size_scale(k->t_uniform), d_c);
    double* qd = q_dev ? q_out : d_q;
    if (small) {
      e = launch_dependent(marginal_small_kernel, dim3(batch), kMargThreads, 16 * ((size_t)1 << std::max(kk - 1, 0)), st, kk,
                           B, k->m, d_x, sizes, coef, qd);
      if (e != cudaSuccess) { ret = cuda_fail(e, "marginal kernel"); break; }
    } else {
      std::vector<int> idx, nv;
      std::vector<int64_t> offs;
      for (int64_t b0 = 0; b0 < batch && ret == GBS_OK; b0 += group) {
        const int cnt = (int)std::min<int64_t>(group, batch - b0);
        if (list) {
          idx.clear();
          nv.clear();
          offs.clear();
          for (int b = 0; b < cnt; ++b)
            for (int c = 0; c < rho.ncls; ++c) {  // every set of the class in colex order
              const int s = rho.t[c];
              unsigned T = (1u << s) - 1;
              for (int64_t r = rho.start[c]; r < rho.start[c + 1]; ++r) {
                offs.push_back((int64_t)idx.size());
                nv.push_back(s);
                for (int i = 0; i < kk; ++i)
                  if (T >> i & 1u) idx.push_back(hx[(size_t)(b0 + b) * kk + i]);
                const unsigned low = T & (0u - T), v = T + low;
                if (low) T = v | (((v ^ T) / low) >> 2);
              }
            }
          if (idx.empty()) idx.push_back(0);
          BatchArgs a;
          a.mode = BatchArgs::PROB;
          a.B = (const double*)B;
          a.m = k->m;
          a.log_norm_dev = k->dscal;
          a.idx = idx.data();
          a.n = nv.data();
          a.offs = offs.data();
          a.batch = (int)nv.size();
          a.precision = GBS_FP64;
          a.stream = st;
          a.out2 = (double*)d_H;
          if ((ret = run_batch(a)) != GBS_OK) break;
        } else {
          for (int s = 0; s <= top; s += 2) {
            const int64_t work = cnt * choose(kk, s);
            marginal_layer_kernel<<<(int)std::min<int64_t>(8192, (work + kMargThreads - 1) / kMargThreads), kMargThreads,
                                    0, st>>>(kk, s, B, k->m, d_x + b0 * kk, cnt, d_H);
          }
        }
        marginal_sum_kernel<<<cnt, kMargThreads, 0, st>>>(kk, rho, list, d_x + b0 * kk, d_H, stride, coef, qd + b0);
      }
      if (ret != GBS_OK) break;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) {
      ret = cuda_fail(e, "marginal kernels");
      break;
    }
    if (!q_dev) {
      e = cudaMemcpyAsync(q_out, d_q, 8 * (size_t)batch, cudaMemcpyDeviceToHost, st);
      if (e == cudaSuccess) e = cudaStreamSynchronize(st);
      if (e != cudaSuccess) {
        ret = cuda_fail(e, "marginal result copy");
        break;
      }
    }
  } while (0);
  scratch_free(tmp, st);
  return ret;
}

// Algorithm 1 for `samples` independent samples at once: x_k of each drawn
// from its m conditional weights q_n(x_1..x_{k-1}, l), l = 0..m-1, with its
// own uniform number (inverse CDF in mode order). A step is three launches
// over all samples (the sums that every candidate shares, the candidates'
// weights, the draw with the cache update), and the steps run without a host
// synchronisation; the modes come back once per group of samples. Groups keep
// their caches within 2^27 entries (2 GB).
extern "C" int gbs_sample_chain_batch(const gbs_kernel* k, int n, int samples, const double* uniforms, void* stream,
                                      int* x_out) {
  clear_error();
  if (!k || (n > 0 && samples > 0 && (!uniforms || !x_out))) return fail(GBS_EINVAL, "null argument");
  if (samples < 0) return fail(GBS_EINVAL, "samples = %d is negative", samples);
  if (n < 0 || n > kMaxK || (n & 1)) return fail(GBS_ERANGE, "n = %d must be even and <= %d", n, kMaxK);
  if (n == 0 || samples == 0) return GBS_OK;
  if (!k->r_uniform) return fail(GBS_EINVAL, "marginals need identical squeezing on every mode");
  if (!(k->t_uniform > 0.0)) return fail(GBS_EINVAL, "marginals need r > 0");
  cudaStream_t st = (cudaStream_t)stream;
  const int m = k->m;
  const int group = std::min({samples, std::max(1, (1 << 28) >> n), 65535});
  auto al = [](size_t v) { return (v + 255) & ~(size_t)255; };
  const int64_t cstride = (int64_t)1 << (n - 1);
  // the steps, last first: what a step reads of the sets that earlier ones add
  std::vector<ChainStep> steps(n + 1);
  unsigned later = 0;
  int tasks = 0;
  for (int kk = n; kk >= 1; --kk) {
    steps[kk] = chain_step(kk, n, m, later);
    tasks = std::max(tasks, steps[kk].tasks);
    const unsigned sizes = rho_sizes(kk, n);
    // rho itself, rho without its new photon and one more, and the sets that
    // the new sets of this step are expanded from
    later |= sizes | (sizes >> 2) | (later >> 2);
  }
  const size_t cache_b = al(16 * (size_t)(group * cstride)), x_b = al(4 * (size_t)group * kMaxK);
  const size_t c_b = al(8 * (size_t)(kMaxK + 1) * kCoefs), q_b = al(8 * (size_t)group * m);
  const size_t part_b = al(16 * (size_t)group * tasks), u_b = al(8 * (size_t)group * n), B_b = al(b_copy_bytes(k));
  void* tmp = nullptr;
  cudaError_t e = scratch_alloc(&tmp, cache_b + x_b + c_b + q_b + part_b + u_b + B_b, st);
  if (e != cudaSuccess) return fail(GBS_ENOMEM, "chain scratch: %s", cudaGetErrorString(e));
  unsigned char* t = (unsigned char*)tmp;
  double2* d_cache = (double2*)t;
  int* d_x = (int*)(t += cache_b);
  double* d_c = (double*)(t += x_b);
  double* d_q = (double*)(t += c_b);
  double2* d_part = (double2*)(t += q_b);
  double* d_u = (double*)(t += part_b);
  const double2* B = (const double2*)scaled_B(k, t + u_b, st);
  std::vector<int> hx((size_t)group * kMaxK);
  int ret = GBS_OK;
  coef_kernel<<<n, kMargThreads, 0, st>>>(1, n, m, size_scale(k->t_uniform), d_c);
  if ((e = cudaGetLastError()) != cudaSuccess) ret = cuda_fail(e, "chain coefficients");
  for (int s0 = 0; s0 < samples && ret == GBS_OK; s0 += group) {
    const int S = std::min(group, samples - s0);
    chain_init_kernel<<<(S + 255) / 256, 256, 0, st>>>(d_cache, cstride, S);
    if ((e = cudaGetLastError()) != cudaSuccess ||
        (e = cudaMemcpyAsync(d_u, uniforms + (size_t)s0 * n, 8 * (size_t)S * n, cudaMemcpyHostToDevice, st)) !=
            cudaSuccess) {
      ret = cuda_fail(e, "chain setup");
      break;
    }
    for (int kk = 1; kk <= n; ++kk) {
      const ChainStep& C = steps[kk];
      constexpr int wpb = kMargThreads / 32;
      e = launch_dependent(chain_gram_kernel, dim3((C.tasks + wpb - 1) / wpb, S), kMargThreads, 0, st, C, d_cache, cstride,
                           B, d_x, d_c, d_part);
      if (e == cudaSuccess)
        e = launch_dependent(chain_weight_kernel, dim3((m + kWeightThreads - 1) / kWeightThreads, S), kWeightThreads, 0, st,
                             C, d_cache, cstride, B, d_x, d_c, d_part, d_q);
      // the draws, then the chosen modes' new sub-Hafnians into the caches
      const int nb = kk < n ? (int)std::max<int64_t>(1, std::min<int64_t>(64, (C.grow.total() + 255) / 256)) : 1;
      if (e == cudaSuccess)
        e = launch_dependent(chain_pick_kernel, dim3(nb, S), kMargThreads, 0, st, C, d_q, d_u, d_x, d_cache, cstride, B);
      if (e != cudaSuccess) break;
    }
    if (e != cudaSuccess) {
      ret = cuda_fail(e, "chain kernels");
      break;
    }
    if ((e = cudaMemcpyAsync(hx.data(), d_x, 4 * (size_t)S * kMaxK, cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess) {
      ret = cuda_fail(e, "chain samples");
      break;
    }
    for (int s = 0; s < S; ++s)
      for (int i = 0; i < n; ++i) x_out[(size_t)(s0 + s) * n + i] = hx[(size_t)s * kMaxK + i];
  }
  scratch_free(tmp, st);
  return ret;
}

// One sample: the batch of one.
extern "C" int gbs_sample_chain(const gbs_kernel* k, int n, const double* uniforms, void* stream, int* x_out) {
  return gbs_sample_chain_batch(k, n, 1, uniforms, stream, x_out);
}

namespace {

// Step 1 of Sec. 3: n from P_n truncated at n_max (renormalised) by the inverse
// CDF with the uniform u.
int pick_photon_number(const std::vector<double>& Pn, int n_max, double tot, double u) {
  const double target = u * tot;
  double run = 0.0;
  for (int v = 0; v <= n_max; v += 2) {
    run += std::max(Pn[v], 0.0);
    if (run > target) return v;
  }
  return n_max & ~1;
}

// P_n for n = 0..n_max and the total of its even entries (GBS_EINVAL if 0).
int truncated_pn(const gbs_kernel* k, int n_max, void* stream, std::vector<double>& Pn, double& tot) {
  Pn.assign((size_t)n_max + 1, 0.0);
  const int rc = gbs_photon_number_dist(k, n_max, stream, Pn.data());
  if (rc) return rc;
  tot = 0.0;
  for (int v = 0; v <= n_max; v += 2) tot += std::max(Pn[v], 0.0);
  if (!(tot > 0.0)) return fail(GBS_EINVAL, "P_n vanishes for every n <= n_max");
  return GBS_OK;
}

}  // namespace

// Steps 1-3 of Sec. 3: n from P_n (truncated at n_max, renormalised) by the
// inverse CDF with uniforms[0], then the chain rule for the n photons.
extern "C" int gbs_sample(const gbs_kernel* k, int n_max, const double* uniforms, void* stream, int* n_out,
                          int* x_out) {
  clear_error();
  if (!k || !uniforms || !n_out || (n_max > 0 && !x_out)) return fail(GBS_EINVAL, "null argument");
  if (n_max < 0 || n_max > kMaxK) return fail(GBS_ERANGE, "n_max = %d outside [0, %d]", n_max, kMaxK);
  if (!k->r_uniform) return fail(GBS_EINVAL, "sampling needs identical squeezing on every mode");
  std::vector<double> Pn;
  double tot = 0.0;
  int rc = truncated_pn(k, n_max, stream, Pn, tot);
  if (rc) return rc;
  const int n = pick_photon_number(Pn, n_max, tot, uniforms[0]);
  *n_out = n;
  if (n == 0) return GBS_OK;
  return gbs_sample_chain(k, n, uniforms + 1, stream, x_out);
}

// gbs_sample for `samples` samples at once: each draws its n, then the samples
// of each n run as one gbs_sample_chain_batch.
extern "C" int gbs_sample_batch(const gbs_kernel* k, int n_max, int samples, const double* uniforms, void* stream,
                                int* n_out, int* x_out) {
  clear_error();
  if (!k || (samples > 0 && (!uniforms || !n_out || (n_max > 0 && !x_out)))) return fail(GBS_EINVAL, "null argument");
  if (samples < 0) return fail(GBS_EINVAL, "samples = %d is negative", samples);
  if (n_max < 0 || n_max > kMaxK) return fail(GBS_ERANGE, "n_max = %d outside [0, %d]", n_max, kMaxK);
  if (!k->r_uniform) return fail(GBS_EINVAL, "sampling needs identical squeezing on every mode");
  if (samples == 0) return GBS_OK;
  std::vector<double> Pn;
  double tot = 0.0;
  int rc = truncated_pn(k, n_max, stream, Pn, tot);
  if (rc) return rc;
  const size_t row = (size_t)n_max + 1;
  std::vector<std::vector<int>> by_n((size_t)n_max + 1);
  for (int s = 0; s < samples; ++s) {
    const int n = pick_photon_number(Pn, n_max, tot, uniforms[s * row]);
    n_out[s] = n;
    by_n[n].push_back(s);
    for (int i = 0; i < n_max; ++i) x_out[(size_t)s * n_max + i] = -1;
  }
  for (int n = 2; n <= n_max; n += 2) {
    const std::vector<int>& idx = by_n[n];
    if (idx.empty()) continue;
    std::vector<double> u(idx.size() * n);
    std::vector<int> x(idx.size() * n);
    for (size_t j = 0; j < idx.size(); ++j)
      for (int i = 0; i < n; ++i) u[j * n + i] = uniforms[idx[j] * row + 1 + i];
    if ((rc = gbs_sample_chain_batch(k, n, (int)idx.size(), u.data(), stream, x.data())) != GBS_OK) return rc;
    for (size_t j = 0; j < idx.size(); ++j)
      for (int i = 0; i < n; ++i) x_out[(size_t)idx[j] * n_max + i] = x[j * n + i];
  }
  return GBS_OK;
}
