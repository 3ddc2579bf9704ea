// sum_S |f(X A_S)|_1 of the subset sum (included by haf_subsets.cu, inside its
// anonymous namespace).
//
// The estimate of a result's error needs the moduli of the subset sum's terms
// f(X A_S) = [x^h] det(I - x X A_S)^{-1/2}; the Hafnian itself comes from the
// matchings (match.cu). For p the last pair of S and S' = S \ {p}, the Schur
// complement of the pairs of S' leaves a 2 x 2 determinant:
//     det(I - x X A_S) = det(I - x X A_S') D_S,   D_S = (1 - b)^2 - a c,
// a, b, c the power series of the walks from p to p whose inside lies in S',
//     b = x A(2p, 2p+1) + sum_k x^{k+2} u^T X (A_S' X)^k v   (a: u u, c: v v),
// u, v the columns 2p and 2p+1 of A on the rows of S'. A term then costs the
// Krylov vectors u_j = (A_S' X)^j u, j <= (h-1)/2, of two columns (walks of
// length i + j from u_i and u_j), about h/2 steps of (2|S'|)^2 products each,
// and three series products, instead of the powers of a 2|S| matrix: 450
// complex multiply-adds against 1500 at n = 16, 3300 against 14,000 at n = 30.
// A and its subsets share one copy in shared memory; a subset keeps vectors
// only, so enough warps are resident to hide latency.
//   terms_delta_kernel   D_S of every subset,
//   terms_series_kernel  f_S = [x^h] prod over the pairs of S of D^{-1/2},
//                        by the last pair: G_S = G_S' D_S^{-1/2}.
// 4096 patterns of n = 16: 0.89 and 0.25 ms (powers in the same arithmetic:
// 2.35 ms and 0.16 for pair sums); 80 of n = 28 and 30, half each: 9.7 and 1.2
// ms (40). The first kernel is bound by issue (0.78 instructions a clock and
// quarter; 20 to 24 warps an SM at n = 28 instead of 16 gave 0.6 %); three
// quarters of its lanes have a row.
//
// Arithmetic. A vector entry is fixed point, (hi + lo) 2^{E_k - 27}, hi a whole
// number of at most 2^27, lo a float of at most a half, with one exponent E_k
// per matrix and power. A complex multiply-add is then 3 IMAD.WIDE (hi hi:
// re re, im im and (re + im)(re + im), summed exactly in 64 bits) and 8 FFMA
// (hi lo and lo hi, which need 24 bits only), instead of 4 DFMA: 28 clocks of
// a warp and SM quarter instead of 256 on this part (DFMA 2 a clock and SM;
// IMAD.WIDE 32; FFMA 128). With four IMAD.WIDE, 80 matrices of n = 28 and 30
// took 19.5 ms instead of 19.0 (n = 16 the same: it is bound by issue); with lo
// an integer too, 52 clocks. The series run in
// pairs of floats (48 FP32 operations a multiply-add), coefficient k in units
// of 2^{e k}, e a mean growth of the E_k.
//
// E_k is fixed per matrix from its full powers (in float, prep kernel) with a
// factor 4..8 of room; an entry is then rounded at 2^-49 of the range. What
// that cannot promise is checked: a value past the range, inputs that are not
// finite, exponents too far apart, or an estimate of the rounding carried along
// with the series (several times what is met, and added over the subsets
// without regard to sign) that comes out above 2^-33 of the sum, send the
// matrix to the FP64 kernels (haf_terms64.cuh; launched after, they return at
// once when no matrix is left to them).
//
// Where this keeps fewer bits than FP64 did, for the estimate alone: a vector
// entry has 2^-49 of its matrix's range, so a small one fewer of its own; D_S,
// its root and G_S are pairs of floats, about 48 bits; a matrix is accepted up
// to a rounding of 2^-33 by an estimate that takes its shares for independent.
// Measured (haf_terms64.cuh), sum |f| is off by 2e-15 as a rule and 4e-14 at
// most, where FP64 had 5e-16; kappa and err_est, its quotients by |Haf|, are
// nearer to their values than before from order 12 on, because the Hafnian is.

constexpr int kFxBits = 27;      // |hi| <= 2^27
constexpr int kFxRoom = 2;       // exponents added to the float estimate of a power's largest entry
constexpr int kExpStride = kExpInts;  // per matrix: E_1, E_2, .. at 1, 2, ..; e at kExpUnit
constexpr int kExpUnit = 18;

// A stored complex entry: x, y = hi (re, im), z, w = lo (float bits). In
// registers hi comes as a float too, for the products with lo. (Cut to its top
// 22 bits, which an addition converts, it cost the estimate of one 16-photon
// pattern four bits.)
struct FxOp {
  int hr, hi, hs;
  float lr, li, fr, fi;
};
__device__ __forceinline__ FxOp fx_load(const int4& v) {
  FxOp o;
  o.hr = v.x;
  o.hi = v.y;
  o.hs = v.x + v.y;
  o.lr = __int_as_float(v.z);
  o.li = __int_as_float(v.w);
  o.fr = (float)v.x;
  o.fi = (float)v.y;
  return o;
}
// One complex sum: h + m, the whole part as sums of re re, im im and
// (re + im)(re + im) (below 2^61: 28 terms of 2^56).
struct Fx {
  long long p, q, s;
  float rm, im;
  __device__ __forceinline__ long long rh() const { return p - q; }
  __device__ __forceinline__ long long ih() const { return s - p - q; }
};
// c += a b
__device__ __forceinline__ void fx_mac(Fx& c, const FxOp& a, const FxOp& b) {
  c.p = (long long)a.hr * b.hr + c.p;
  c.q = (long long)a.hi * b.hi + c.q;
  c.s = (long long)a.hs * b.hs + c.s;
  c.rm = fmaf(a.fr, b.lr, c.rm);
  c.im = fmaf(a.fr, b.li, c.im);
  c.rm = fmaf(-a.fi, b.li, c.rm);
  c.im = fmaf(a.fi, b.lr, c.im);
  c.rm = fmaf(a.lr, b.fr, c.rm);
  c.im = fmaf(a.lr, b.fi, c.im);
  c.rm = fmaf(-a.li, b.fi, c.rm);
  c.im = fmaf(a.li, b.fr, c.im);
}
__device__ __forceinline__ Fx fx_zero() { return Fx{0, 0, 0, 0.0f, 0.0f}; }
// (hi, lo) = hi + lo with |lo| <= 1/2 (|lo| < 2^22 before); over where |hi| > 2^27.
__device__ __forceinline__ int2 fx_pack(int hi, float lo, bool& over) {
  const float q = lo + 12582912.0f;
  hi += __float_as_int(q) - 0x4B400000;
  over |= (unsigned)(hi + (1 << kFxBits)) > (2u << kFxBits);
  return make_int2(hi, __float_as_int(lo - (q - 12582912.0f)));
}
// (h + m) 2^-sh, 18 <= sh <= 31 (so h 2^-sh is below 2^44).
__device__ __forceinline__ int2 fx_round(long long h, float m, int sh, bool& over) {
  const long long top = h >> sh;
  over |= (unsigned)((int)(top >> 28) + 1) > 1u || !(fabsf(m) < 0x1p36f);
  const float unit = __int_as_float((127 - sh) << 23);
  const float lo = (float)((unsigned)h & ((1u << sh) - 1)) * unit + m * unit;
  return fx_pack((int)top, lo, over);
}
__device__ __forceinline__ int4 fx_entry(const Fx& c, int sh, bool& over) {
  const int2 x = fx_round(c.rh(), c.rm, sh, over), y = fx_round(c.ih(), c.im, sh, over);
  return make_int4(x.x, y.x, x.y, y.y);
}
__device__ __forceinline__ bool fx_shift_ok(int sh) { return sh >= 18 && sh <= 31; }


// Per matrix: the exponents, the entries' limbs (rows and columns in the
// subset sum's order, zero diagonal), and whether it can be done in fixed
// point at all. One block per matrix. The powers of the whole matrix, scaled
// to entries below 1, are formed in float only for the size of their largest
// entry.
__global__ void __launch_bounds__(256) terms_prep_kernel(const TermsLaunch P, const TermsChunk C) {
  __shared__ float2 A[kMaxN * kMaxN], R[kMaxN * kMaxN];
  __shared__ int rows[kMaxN], s_max[kMaxN / 2 + 1], s_lo, s_bad;
  dependency_wait();
  int g = 0;
  while (g + 1 < C.n_groups && (int)blockIdx.x >= C.g[g + 1].begin) ++g;
  const TermsGroup G = C.g[g];
  const int q = blockIdx.x - G.begin, b = P.order[G.first + q];
  const PatDesc d = P.pats[b];
  const int n = G.n, h = n >> 1;
  if (P.skip != nullptr && P.skip[b] != 0) return;
  if (threadIdx.x < n) {
    int pos = default_pos(threadIdx.x, h);
    if (P.perm != nullptr && P.perm_off[b] >= 0) pos = P.perm[P.perm_off[b] + threadIdx.x];
    int v = (d.idx_off >= 0) ? P.idx[d.idx_off + pos] : pos;
    if (P.m_bound > 0 && (v < 0 || v >= P.m_bound)) {
      P.status[b] = 1;
      v = 0;
    }
    rows[threadIdx.x] = v;
  }
  if (threadIdx.x <= kMaxN / 2) s_max[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    s_bad = 0;
    s_lo = 0x7fffffff;
  }
  __syncthreads();
  const double2* src2 = reinterpret_cast<const double2*>(P.src) + d.src_off;
  // largest binary exponent (0: zero or subnormal, 2047: not finite) of the
  // matrix, and the smallest of its rows' largest ones
  int mine = 0;
  for (int r = threadIdx.x >> 5; r < n; r += blockDim.x >> 5) {
    const int c = threadIdx.x & 31;
    int e = 0;
    if (c < n && c != r) {
      const double2 v = __ldg(src2 + (int64_t)rows[min(r, c)] * d.ld + rows[max(r, c)]);
      e = max((__double2hiint(v.x) >> 20) & 2047, (__double2hiint(v.y) >> 20) & 2047);
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (c == 0) {
      mine = max(mine, e);
      atomicMin(&s_lo, e);
    }
  }
  if ((threadIdx.x & 31) == 0) atomicMax(&s_max[0], mine);
  __syncthreads();
  const int e1 = s_max[0] - 1022;  // every |entry| < 2^e1
  // rows more than 2^20 apart in size would lose bits next to each other
  if (e1 > 900 || e1 < -900 || s_max[0] - s_lo > 20) return;  // ok stays 0 (uniform)
  const double up = __hiloint2double((kFxBits - e1 + 1023) << 20, 0);
  const double unit = __hiloint2double((1023 - e1) << 20, 0);
  int4* out = reinterpret_cast<int4*>(C.scratch) + G.off + (int64_t)q * G.stride;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int r = e / n, c = e - r * n;
    double2 v = make_double2(0.0, 0.0);
    if (r != c) v = __ldg(src2 + (int64_t)rows[min(r, c)] * d.ld + rows[max(r, c)]);
    A[e] = R[e] = make_float2((float)(v.x * unit), (float)(v.y * unit));
    const double x = v.x * up, y = v.y * up;
    const int hx = __double2int_rn(x), hy = __double2int_rn(y);
    out[e] = make_int4(hx, hy, __float_as_int((float)(x - hx)), __float_as_int((float)(y - hy)));
  }
  __syncthreads();
  // largest entries of the powers that vectors reach, as float bits
  const int top = (h + 1) / 2;
  for (int k = 2; k <= top; ++k) {
    float2 acc[4];
    float big = 0.0f;
    int i = 0;
    for (int e = threadIdx.x; e < n * n; e += blockDim.x, ++i) {
      const int r = e / n, c = e - r * n;
      float2 s = make_float2(0.f, 0.f);
      for (int t = 0; t < n; ++t) {
        const float2 x = R[r * n + t], y = A[(t ^ 1) * n + c];
        s.x = fmaf(x.x, y.x, s.x);
        s.x = fmaf(-x.y, y.y, s.x);
        s.y = fmaf(x.x, y.y, s.y);
        s.y = fmaf(x.y, y.x, s.y);
      }
      acc[i] = s;
      big = fmaxf(big, fmaxf(fabsf(s.x), fabsf(s.y)));
    }
    atomicMax(&s_max[k], __float_as_int(big));
    __syncthreads();
    i = 0;
    for (int e = threadIdx.x; e < n * n; e += blockDim.x, ++i) R[e] = acc[i];
    __syncthreads();
  }
  int* ex = P.exps + (int64_t)b * kExpStride;
  if (threadIdx.x >= 1 && (int)threadIdx.x <= top) {
    const int k = threadIdx.x;
    int ek = e1;
    for (int j = 2; j <= k; ++j) {
      const int f = (s_max[j] >> 23) & 255;
      if (f < 20 || f > 250) s_bad = 1;  // zero, vanishing or not finite
      // a step's rounding shifts by 31 bits at most: where a power grows by
      // more, its range gets less room instead (one matrix in 2e4 of 16 modes
      // out of 64 went to the FP64 kernels for it)
      ek = min(j * e1 + f - 126 + kFxRoom, ek + e1 + 4);
    }
    ex[k] = ek;
    if (k == top) ex[kExpUnit] = __float2int_rn((float)ek / (float)top);
  }
  __syncthreads();
  if (threadIdx.x == 0 && !s_bad) P.ok[b] = 1;
}

// ---- pairs of floats ------------------------------------------------------
// A complex number: x, y = high parts (re, im), z, w = low parts.
// s += a b of one component; the low sum gathers every rounding error but its
// own (Dekker and Knuth; no contraction between the steps).
__device__ __forceinline__ void df_mac(float& sh, float& sl, float ah, float al, float bh, float bl) {
  const float p = __fmul_rn(ah, bh);
  float e = __fmaf_rn(ah, bh, -p);
  e = __fmaf_rn(ah, bl, e);
  e = __fmaf_rn(al, bh, e);
  const float s = __fadd_rn(sh, p), z = __fsub_rn(s, sh);
  const float w = __fadd_rn(__fsub_rn(sh, __fsub_rn(s, z)), __fsub_rn(p, z));
  sh = s;
  sl = __fadd_rn(sl, __fadd_rn(w, e));
}
__device__ __forceinline__ void dfc_mac(float4& c, const float4& a, const float4& b) {
  df_mac(c.x, c.z, a.x, a.z, b.x, b.z);
  df_mac(c.y, c.w, a.x, a.z, b.y, b.w);
  df_mac(c.x, c.z, -a.y, -a.w, b.y, b.w);
  df_mac(c.y, c.w, a.y, a.w, b.x, b.z);
}
__device__ __forceinline__ float4 dfc_norm(const float4& c) {
  const float h = __fadd_rn(c.x, c.z), i = __fadd_rn(c.y, c.w);
  return make_float4(h, i, __fsub_rn(c.z, __fsub_rn(h, c.x)), __fsub_rn(c.w, __fsub_rn(i, c.y)));
}
// a times a float (exactly rounded at the low part).
__device__ __forceinline__ float4 dfc_scale(const float4& a, float f) {
  const float x = __fmul_rn(a.x, f), y = __fmul_rn(a.y, f);
  return make_float4(x, y, __fmaf_rn(a.z, f, __fmaf_rn(a.x, f, -x)), __fmaf_rn(a.w, f, __fmaf_rn(a.y, f, -y)));
}
__device__ __forceinline__ float dfc_abs1(const float4& a) { return fabsf(a.x) + fabsf(a.y); }
// (h + m) unit as a pair of floats, |h| < 2^61: the top 31 and the low 30 bits,
// each as a float and what that leaves, by 32-bit conversions (64-bit ones run
// on the FP64 pipe, which they held a quarter of the time).
__device__ __forceinline__ float2 df_from(long long h, float m, float unit) {
  const int a = (int)(h >> 30), r = (int)h & 0x3fffffff;
  const float fa = (float)a, fr = (float)r, hi = fa * 0x1p30f;
  const float rest = __fadd_rn((float)(a - (int)fa) * 0x1p30f, __fadd_rn((float)(r - (int)fr), m));
  const float t = __fadd_rn(hi, fr);  // (|hi| >= 2^30 > fr, or hi = 0)
  const float lo = __fadd_rn(__fsub_rn(fr, __fsub_rn(t, hi)), rest);
  const float s = __fadd_rn(t, lo);
  return make_float2(s * unit, __fsub_rn(lo, __fsub_rn(s, t)) * unit);
}
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }  // -126 <= e <= 127

// D_S of every subset: a warp takes rounds of 32 / L subsets of one size, L
// lanes each (lane = row of S'; then one of the 3 (h - 1) sums; then one
// coefficient). Round r of a matrix: the sizes in order, the subsets of a size
// in colex order, consecutive ones side by side. Block (matrix, part) has
// rounds part, part + parts, ..
__global__ void __launch_bounds__(kDeltaThreads) terms_delta_kernel(const TermsLaunch P, const TermsChunk C) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int binom[kMaxH + 1][kMaxH + 1], ex[kExpStride], s_bad;
  __shared__ float unit[kMaxH + 1];  // of the coefficient x^k, k >= 2
  if (threadIdx.x <= kMaxH) {
    const int a = threadIdx.x;
    int c = 1;
    for (int b = 0; b <= kMaxH; ++b) {  // C(a, b) = C(a, b-1) (a-b+1) / b
      binom[a][b] = (b <= a) ? c : 0;
      if (b < a) c = c * (a - b) / (b + 1);
    }
  }
  if (threadIdx.x == 0) s_bad = 0;
  dependency_wait();
  int g = 0;
  while (g + 1 < C.n_groups && (int)blockIdx.x >= C.g[g + 1].block) ++g;
  const TermsGroup G = C.g[g];
  const int n = G.n, h = n >> 1, q = (blockIdx.x - G.block) / G.parts, part = (blockIdx.x - G.block) - q * G.parts;
  const int b = P.order[G.first + q];
  if (P.ok[b] == 0) return;  // uniform (no block writes it here): not in fixed point, or the repeated-row sum's
  const int4* mat = reinterpret_cast<const int4*>(C.scratch) + G.off + (int64_t)q * G.stride;
  float4* delta = reinterpret_cast<float4*>(const_cast<int4*>(mat) + n * n);
  int4* M = reinterpret_cast<int4*>(smem);
  const int ld = n + 1;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int r = e / n;
    M[r * ld + e - r * n] = mat[e];
  }
  if (threadIdx.x < kExpStride) ex[threadIdx.x] = P.exps[(int64_t)b * kExpStride + threadIdx.x];
  __syncthreads();
  const int steps = (h - 1) / 2;  // vectors u_0 .. u_steps
  if (threadIdx.x >= 1 && (int)threadIdx.x <= steps) {
    const int k = threadIdx.x;
    if (!fx_shift_ok(27 + ex[k + 1] - ex[k] - ex[1])) s_bad = 1;
  }
  if (threadIdx.x >= 1 && (int)threadIdx.x <= h) {
    const int k = threadIdx.x, i = (k - 2) >> 1;
    // x^1: the entry itself; x^k: u_i and u_j, i + j = k - 2, exponents E_{i+1}, E_{j+1}
    const int e = (k == 1) ? ex[1] - 27 - ex[kExpUnit] : ex[i + 1] + ex[k - 2 - i + 1] - 54 - k * ex[kExpUnit];
    if (e < -120 || e > 0) s_bad = 1;
    unit[k] = pow2f(max(min(e, 120), -120));
  }
  __syncthreads();
  if (s_bad) {
    if (threadIdx.x == 0) P.lost[b] = 1;
    return;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  unsigned char* wbase = smem + (size_t)n * ld * 16 + (size_t)warp * G.region;
  bool over = false;
  int s = 1, done = 0;  // rounds of the sizes below s
  for (int r = part * nw + warp;; r += G.parts * nw) {
    int L = terms_lanes(s), rounds = (binom[h][s] + 32 / L - 1) / (32 / L);
    while (r - done >= rounds) {
      done += rounds;
      if (++s > h) break;
      L = terms_lanes(s);
      rounds = (binom[h][s] + 32 / L - 1) / (32 / L);
    }
    if (s > h) break;
    const int gpw = 32 / L, gi = min(lane / L, gpw - 1), l = lane - gi * L;  // lanes past the last group: l >= L
    const int rank = (r - done) * gpw + gi;
    const bool active = rank < binom[h][s] && l < L;
    int4* V = reinterpret_cast<int4*>(wbase + (size_t)gi * terms_group_bytes(s, h));
    const int sp = s - 1, N = 2 * sp;
    float4* mom = reinterpret_cast<float4*>(V + (steps + 1) * 2 * N);  // a, b, c at 3 (k - 1) + 0, 1, 2
    int* pairs = reinterpret_cast<int*>(mom + 3 * h);
    unsigned mask = 0;
    {
      int rk = min(rank, binom[h][s] - 1), c = h - 1;
      for (int i = s; i >= 1; --i) {
        while (binom[c][i] > rk) --c;
        rk -= binom[c][i];
        mask |= 1u << c;
        --c;
      }
    }
    const int p = 31 - __clz((int)mask);
    const unsigned rest = mask ^ (1u << p);
    if (l < sp) {
      unsigned m = rest;
      for (int t = 0; t < l; ++t) m &= m - 1;
      pairs[l] = __ffs((int)m) - 1;
    }
    __syncwarp();
    const bool mine = l < N;
    const int4* row = M + (mine ? 2 * pairs[l >> 1] + (l & 1) : 0) * ld;
    if (mine) {
      V[l] = row[2 * p];
      V[N + l] = row[2 * p + 1];
    }
    __syncwarp();
    for (int k = 1; k <= steps; ++k) {
      if (mine) {
        const int4* U = V + (k - 1) * 2 * N;
        Fx ca = fx_zero(), cb = ca;
#pragma unroll 1
        for (int t = 0; t < sp; ++t) {
          const int c = 2 * pairs[t];
          const FxOp x0 = fx_load(row[c]), x1 = fx_load(row[c + 1]);
          const FxOp a1 = fx_load(U[2 * t + 1]), a0 = fx_load(U[2 * t]);
          const FxOp b1 = fx_load(U[N + 2 * t + 1]), b0 = fx_load(U[N + 2 * t]);
          fx_mac(ca, x0, a1);
          fx_mac(cb, x0, b1);
          fx_mac(ca, x1, a0);
          fx_mac(cb, x1, b0);
        }
        const int sh = 27 + ex[k + 1] - ex[k] - ex[1];
        V[k * 2 * N + l] = fx_entry(ca, sh, over);
        V[k * 2 * N + N + l] = fx_entry(cb, sh, over);
      }
      __syncwarp();
    }
    // the walks' sums, one a lane; the three of x^1, which cost nothing, last
    for (int r1 = l; l < L && r1 < 3 * h; r1 += L) {
      const int t = 3 * h - 1 - r1, k = t / 3 + 1, type = t - 3 * (k - 1);
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (k == 1) {
        if (type == 1) {
          const int4 e = M[2 * p * ld + 2 * p + 1];
          const float u = unit[1];
          const float hr = (float)e.x, hi = (float)e.y;
          v = dfc_norm(make_float4(hr * u, hi * u, ((float)(e.x - (int)hr) + __int_as_float(e.z)) * u,
                                   ((float)(e.y - (int)hi) + __int_as_float(e.w)) * u));
        }
      } else {
        const int i = (k - 2) >> 1, j = k - 2 - i;
        const int4* x = V + i * 2 * N + (type == 2 ? N : 0);
        const int4* y = V + j * 2 * N + (type == 0 ? 0 : N);
        Fx c = fx_zero();
#pragma unroll 2
        for (int r2 = 0; r2 < N; ++r2) {
          const FxOp xr = fx_load(x[r2]);
          fx_mac(c, xr, fx_load(y[r2 ^ 1]));
        }
        const float2 re = df_from(c.rh(), c.rm, unit[k]), im = df_from(c.ih(), c.im, unit[k]);
        v = make_float4(re.x, im.x, re.y, im.y);
      }
      mom[t] = v;
    }
    __syncwarp();
    // coefficient k of D_S = 1 - 2 b + b^2 - a c, one a lane, the longest first:
    // where there are more than lanes, the second turn has the short ones (with
    // b_i b_(k-i) formed once for both: 1.75 -> 1.69 ms at 4096 x n = 16, 20.0
    // -> 19.4 at 80 of n = 28 and 30)
    for (int r1 = l; l < L && r1 < h; r1 += L) {
      const int k = h - r1;
      float4 c = dfc_scale(mom[3 * (k - 1) + 1], -2.0f);
#pragma unroll 1
      for (int i = 1; i < k; ++i) {
        const float4 ai = mom[3 * (i - 1)];
        dfc_mac(c, make_float4(-ai.x, -ai.y, -ai.z, -ai.w), mom[3 * (k - i - 1) + 2]);
        if (2 * i <= k) {
          const float4 bi = mom[3 * (i - 1) + 1];
          const float f = 2 * i == k ? 1.0f : 2.0f;  // b_i b_(k-i) twice
          dfc_mac(c, make_float4(bi.x * f, bi.y * f, bi.z * f, bi.w * f), mom[3 * (k - i - 1) + 1]);
        }
      }
      if (active) delta[(int64_t)mask * h + k - 1] = dfc_norm(c);
    }
    __syncwarp();
  }
  if (over) P.lost[b] = 1;
}

// The last pair's factor and the product with the subset before, a thread per
// subset. Masks below 256 by one block per matrix, level after level (`level`
// < 0); the masks with last pair `level` >= 8 by 2^level / 256 blocks a matrix.
// A block's sum |f|_1 and its rounding go to parts[mask >> 8].
__global__ void __launch_bounds__(256) terms_series_kernel(const TermsLaunch P, const TermsChunk C, int level) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double red[2][256];
  __shared__ float cn[kMaxH + 1];
  // masks below 256: D_S, then its root, coefficient k of S at [k - 1][S]; the
  // row takes one place more, so that neither the copy (a subset's
  // coefficients side by side) nor the sums (subsets side by side) collide (read
  // from device memory, a place per lane 128 bytes apart, they kept the load
  // pipe 62 % busy; with twice the threads of the matchings' tiles 4096 of
  // n = 16 go from 1.72 to 1.63 ms, 80 of n = 28 and 30 from 18.7 to 18.4)
  float4* ys = reinterpret_cast<float4*>(smem);
  constexpr int ld = 257;
  dependency_wait();
  int g = 0, bid = blockIdx.x;
  const int per = level < 0 ? 1 : 1 << (level - 8);
  for (; g < C.n_groups; ++g) {
    const int blocks = (C.g[g].n >> 1) > level ? C.g[g].count * per : 0;
    if (bid < blocks) break;
    bid -= blocks;
  }
  if (g == C.n_groups) return;
  const TermsGroup G = C.g[g];
  const int n = G.n, h = n >> 1, q = bid / per, sub = bid - q * per, b = P.order[G.first + q];
  if (P.ok[b] == 0 || P.lost[b] != 0) return;
  int4* base = reinterpret_cast<int4*>(C.scratch) + G.off + (int64_t)q * G.stride;
  const float4* delta = reinterpret_cast<const float4*>(base + n * n);
  float4* Gs = reinterpret_cast<float4*>(base + n * n) + ((int64_t)h << h);  // coefficient k of G_S at [k - 1][S], S without pair h - 1
  const int64_t gl = (int64_t)1 << (h - 1);
  double2* parts = reinterpret_cast<double2*>(Gs + gl * h);
  const int* ex = P.exps + (int64_t)b * kExpStride;
  if (threadIdx.x >= 1 && (int)threadIdx.x <= h) {
    // rounding of coefficient k of a, b, c, in its units: up to n products of
    // entries off by 2^-50 of their range, independently, with entries of a
    // quarter of theirs at most (the room): sqrt(n) 2^-51 is several times that
    const int k = threadIdx.x, i = (k - 2) >> 1;
    const int e = (k == 1) ? ex[1] - 48 - ex[kExpUnit] : ex[i + 1] + ex[k - 2 - i + 1] - 51 - k * ex[kExpUnit];
    cn[k] = sqrtf((float)n) * pow2f(max(min(e, 100), -120));
  }
  if (level < 0)
    for (int e = threadIdx.x + h; e < h << min(h, 8); e += blockDim.x) ys[(e % h) * ld + e / h] = delta[e];
  __syncthreads();
  double kap = 0.0, noise = 0.0;
  float4 y[kMaxH];
  // y = D^{-1/2} of the thread's subset: k y_k = -sum_i (k - i / 2) d_i y_{k-i}
  auto root = [&](const float4* d, int step) {
    float4 dl[kMaxH];
#pragma unroll 1
    for (int k = 0; k < h; ++k) dl[k] = d[k * step];
#pragma unroll 1
    for (int k = 1; k <= h; ++k) {
      float4 c = dfc_scale(dl[k - 1], 0.5f * k);  // i = k, y_0 = 1
#pragma unroll 1
      for (int i = 1; i < k; ++i) dfc_mac(c, dfc_scale(dl[i - 1], (float)k - 0.5f * i), y[k - i - 1]);
      // times -1/k as a pair of floats
      const float r = __frcp_rn((float)k), rl = __fmul_rn(__fmaf_rn(-r, (float)k, 1.0f), r);
      float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
      c = dfc_norm(c);
      df_mac(o.x, o.z, c.x, c.z, -r, -rl);
      df_mac(o.y, o.w, c.y, c.w, -r, -rl);
      y[k - 1] = dfc_norm(o);
    }
  };
  // coefficient k of G_S = G_S' y, y's at y[(k - 1) step]; at k = h counts f_S
  // and its rounding
  auto grow = [&](int S, int p, int k, const float4* y, int step) {
    const int Sp = S ^ (1 << p);
    float4 c = y[(k - 1) * step];
    float size = dfc_abs1(c), nz = cn[h];
    if (Sp != 0) {
      const float4* gp = Gs + Sp;
      const float4 t = gp[(k - 1) * gl], one = make_float4(1.f, 0.f, 0.f, 0.f);
      size += dfc_abs1(t);
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
      for (int i = 1; i < k; ++i) {
        const float4 g0 = gp[(i - 1) * gl], y0 = y[(k - i - 1) * step];
        dfc_mac(a, g0, y0);
        size += dfc_abs1(g0) * dfc_abs1(y0);
        if (k == h) nz += cn[k - i] * dfc_abs1(g0);
      }
      dfc_mac(a, one, c);
      dfc_mac(a, one, t);
      c = dfc_norm(a);
    }
    if (p < h - 1) Gs[(k - 1) * gl + S] = c;
    if (k == h) {
      nz += 0x1p-42f * size;  // rounding of the series themselves
      kap += fabs((double)c.x + (double)c.z) + fabs((double)c.y + (double)c.w);
      noise += 4.0 * (double)nz;  // the pairs before this one too: up to 14 independent shares
    }
  };
  if (level < 0) {
    // a thread per subset, then per subset and coefficient of a level
    const int low = min(h, 8);
    if (threadIdx.x >= 1 && (int)threadIdx.x < (1 << low)) {
      root(ys + threadIdx.x, ld);
      for (int k = 0; k < h; ++k) ys[k * ld + threadIdx.x] = y[k];
    }
    for (int p = 0; p < low; ++p) {
      __syncthreads();
      if (p < h - 1) {
        for (int t = threadIdx.x; t < h << p; t += blockDim.x) {
          const int S = (1 << p) + (t & ((1 << p) - 1));
          grow(S, p, h - (t >> p), ys + S, ld);
        }
      } else if ((int)threadIdx.x < (1 << p)) {
        grow((1 << p) + threadIdx.x, p, h, ys + (1 << p) + threadIdx.x, ld);
      }
    }
  } else {
    const int S = (1 << level) + sub * 256 + threadIdx.x;
    root(delta + (int64_t)S * h, 1);
    for (int k = (level < h - 1) ? 1 : h; k <= h; ++k) grow(S, level, k, y, 1);
  }
  red[0][threadIdx.x] = kap;
  red[1][threadIdx.x] = noise;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      red[0][threadIdx.x] += red[0][threadIdx.x + o];
      red[1][threadIdx.x] += red[1][threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) parts[level < 0 ? 0 : per + sub] = make_double2(red[0][0], red[1][0]);
}

// One warp per matrix: the sum over its parts, in its own units again; a matrix
// that left the range, or whose rounding estimate is above 2^-33 of the sum, goes
// to the FP64 kernels.
__global__ void __launch_bounds__(256) terms_check_kernel(const TermsLaunch P, const TermsChunk C) {
  dependency_wait();
  const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  const TermsGroup& last = C.g[C.n_groups - 1];
  const int mats = last.begin + last.count;
  bool redo = false;
  for (int m = blockIdx.x * wpb + (threadIdx.x >> 5); m < mats; m += gridDim.x * wpb) {
    int g = 0;
    while (g + 1 < C.n_groups && m >= C.g[g + 1].begin) ++g;
    const TermsGroup& G = C.g[g];
    const int n = G.n, h = n >> 1, q = m - G.begin, b = P.order[G.first + q];
    if (P.skip != nullptr && P.skip[b] != 0) {
      if (lane == 0) P.ok[b] = 1;  // nothing for the FP64 kernels either
      continue;
    }
    double K = 0.0, noise = 0.0;
    const bool done = P.ok[b] != 0 && P.lost[b] == 0;
    if (done) {
      const int4* base = reinterpret_cast<const int4*>(C.scratch) + G.off + (int64_t)q * G.stride;
      const double2* parts = reinterpret_cast<const double2*>(base + n * n + ((int64_t)h << h) + ((int64_t)h << (h - 1)));
      for (int i = lane; i < (h > 8 ? 1 << (h - 8) : 1); i += 32) {
        K += parts[i].x;
        noise += parts[i].y;
      }
    }
    for (int off = 16; off > 0; off >>= 1) {
      K += __shfl_xor_sync(0xffffffffu, K, off);
      noise += __shfl_xor_sync(0xffffffffu, noise, off);
    }
    if (lane == 0) {
      const bool fine = done && noise <= 0x1p-33 * K && K > 0x1p-90 && K < 0x1p120;
      P.ksum[b] = fine ? ldexp(K, h * P.exps[(int64_t)b * kExpStride + kExpUnit]) : 0.0;
      P.ok[b] = fine ? 1 : 0;
      redo |= !fine;
    }
  }
  if (redo) *P.left = 1;  // (zero before the first chunk; every writer writes the same)
}
