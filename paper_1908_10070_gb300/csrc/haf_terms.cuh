// sum_S |f(X A_S)|_1 of the subset sum, in fixed point (included by
// haf_subsets.cu, inside its anonymous namespace).
//
// The estimate of a result's error needs the moduli of the subset sum's terms;
// the Hafnian itself comes from the matchings (match.cu). The terms' power
// traces are the FP64 kernel's, but a product entry here is fixed point: an
// entry of R_k = A (X A)^{k-1} is (hi + lo) 2^{E_k - 27}, hi a whole number of
// at most 2^27, lo a float of at most a half, with one exponent E_k per matrix
// and power. A complex multiply-add is then 4 IMAD.WIDE (hi hi, summed exactly
// in 64 bits) and 8 FFMA (hi lo and lo hi, which need 24 bits only), instead of
// 4 DFMA: 32 clocks of a warp and SM quarter instead of 256 on this part (DFMA
// 2 a clock and SM; IMAD.WIDE 32; FFMA 128). All four products as IMAD.WIDE,
// with lo an integer too, took 52.
//
// E_k is fixed per matrix from its full powers (in float, prep kernel) with a
// factor 4..8 of room; an entry is then rounded at 2^-49 of the range. What
// that cannot promise is checked: a value past the range, inputs that are not
// finite, exponents too far apart, or a bound on the rounding carried along
// with the series that comes out above 2^-33 of the sum, send the matrix to
// the FP64 kernel (launched after; it returns at once when no matrix is left
// to it).

constexpr int kFxBits = 27;      // |hi| <= 2^27
constexpr int kFxRoom = 2;       // exponents added to the float estimate of a power's largest entry
constexpr int kTermsHeader = 512;  // per warp: scales, rounding bounds, exponents
constexpr int kExpStride = 20;   // exponents kept per matrix
constexpr int kSumBlocks = 8;    // 2 x 2 blocks of pair sums per thread block

// A stored complex entry: x, y = hi (re, im), z, w = lo (float bits). In
// registers hi comes as a float too, hi 2^-6 cut to a whole number (the
// products with lo need no more), by adding and taking off 1.5 2^23.
struct FxOp {
  int hr, hi;
  float lr, li, fr, fi;
};
__device__ __forceinline__ float fx_float(int h) { return __int_as_float((h >> 6) + 0x4B400000) - 12582912.0f; }
__device__ __forceinline__ FxOp fx_load(const int4& v) {
  FxOp o;
  o.hr = v.x;
  o.hi = v.y;
  o.lr = __int_as_float(v.z);
  o.li = __int_as_float(v.w);
  o.fr = fx_float(v.x);
  o.fi = fx_float(v.y);
  return o;
}
struct Fx {  // one complex sum: h + 64 m
  long long rh, ih;
  float rm, im;
};
// c += a b; n = -a.hi
__device__ __forceinline__ void fx_mac(Fx& c, const FxOp& a, int n, const FxOp& b) {
  c.rh = (long long)a.hr * b.hr + c.rh;
  c.ih = (long long)a.hr * b.hi + c.ih;
  c.rm = fmaf(a.fr, b.lr, c.rm);
  c.im = fmaf(a.fr, b.li, c.im);
  c.rh = (long long)n * b.hi + c.rh;
  c.ih = (long long)a.hi * b.hr + c.ih;
  c.rm = fmaf(-a.fi, b.li, c.rm);
  c.im = fmaf(a.fi, b.lr, c.im);
  c.rm = fmaf(a.lr, b.fr, c.rm);
  c.im = fmaf(a.lr, b.fi, c.im);
  c.rm = fmaf(-a.li, b.fi, c.rm);
  c.im = fmaf(a.li, b.fr, c.im);
}
__device__ __forceinline__ Fx fx_zero() { return Fx{0, 0, 0.0f, 0.0f}; }
// (hi, lo) = hi + lo with |lo| <= 1/2 (|lo| < 2^22 before); over where |hi| > 2^27.
__device__ __forceinline__ int2 fx_pack(int hi, float lo, bool& over) {
  const float q = lo + 12582912.0f;
  hi += __float_as_int(q) - 0x4B400000;
  over |= (unsigned)(hi + (1 << kFxBits)) > (2u << kFxBits);
  return make_int2(hi, __float_as_int(lo - (q - 12582912.0f)));
}
// (h + 64 m) 2^-sh, 18 <= sh <= 31 (so h 2^-sh is below 2^44).
__device__ __forceinline__ int2 fx_round(long long h, float m, int sh, bool& over) {
  const long long top = h >> sh;
  over |= (unsigned)((int)(top >> 28) + 1) > 1u || !(fabsf(m) < 0x1p30f);
  const float unit = __int_as_float((127 - sh) << 23);
  const float lo = (float)((unsigned)h & ((1u << sh) - 1)) * unit + m * (64.0f * unit);
  return fx_pack((int)top, lo, over);
}
__device__ __forceinline__ int4 fx_entry(const Fx& c, int sh, bool& over) {
  const int2 x = fx_round(c.rh, c.rm, sh, over), y = fx_round(c.ih, c.im, sh, over);
  return make_int4(x.x, y.x, x.y, y.y);
}
__device__ __forceinline__ bool fx_shift_ok(int sh) { return sh >= 18 && sh <= 31; }

// A symmetric matrix of s pairs as 2 x 2 blocks of its upper block triangle:
// block (r, c), r < c, is number c(c-1)/2 + r, block (r, r) number
// s(s-1)/2 + r; element 2 i + j of a block is entry (2r + i, 2c + j).
__device__ __forceinline__ int blk_index(int r, int c, int s) {
  const int lo = min(r, c), hi = max(r, c);
  return lo == hi ? s * (s - 1) / 2 + lo : hi * (hi - 1) / 2 + lo;
}

// Per matrix: the exponents, the entries' limbs (block layout of all h pairs,
// elements innermost), and whether it can be done in fixed point at all. One
// block per matrix. The powers of the whole matrix, scaled to entries below 1,
// are formed in float only for the size of their largest entry.
__global__ void __launch_bounds__(256) terms_prep_kernel(const TermsLaunch P) {
  __shared__ float2 A[kMaxN * kMaxN], R[kMaxN * kMaxN];
  __shared__ int rows[kMaxN], s_max[kMaxN / 2 + 1], s_lo, s_bad;
  dependency_wait();
  const int b = blockIdx.x;
  const PatDesc d = P.pats[b];
  const int n = d.n, h = n >> 1;
  if (n < 2 || (n & 1) || P.mat_off[b] < 0) return;
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
  int4* out = P.mat + P.mat_off[b];
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    const int r = e / n, c = e - r * n;
    double2 v = make_double2(0.0, 0.0);
    if (r != c) v = __ldg(src2 + (int64_t)rows[min(r, c)] * d.ld + rows[max(r, c)]);
    A[e] = R[e] = make_float2((float)(v.x * unit), (float)(v.y * unit));
    if ((r >> 1) <= (c >> 1)) {
      const double x = v.x * up, y = v.y * up;
      const int hx = __double2int_rn(x), hy = __double2int_rn(y);
      out[4 * blk_index(r >> 1, c >> 1, h) + 2 * (r & 1) + (c & 1)] =
          make_int4(hx, hy, __float_as_int((float)(x - hx)), __float_as_int((float)(y - hy)));
    }
  }
  __syncthreads();
  // largest entries of the powers the schedule keeps, as float bits
  const int top = (int)((0x8877665645332211ull >> (4 * (h - 1))) & 15u);
  for (int k = 2; k <= top; ++k) {
    float2 acc[4];
    float big = 0.0f;
    int q = 0;
    for (int e = threadIdx.x; e < n * n; e += blockDim.x, ++q) {
      const int r = e / n, c = e - r * n;
      float2 s = make_float2(0.f, 0.f);
      for (int t = 0; t < n; ++t) {
        const float2 x = R[r * n + t], y = A[(t ^ 1) * n + c];
        s.x = fmaf(x.x, y.x, s.x);
        s.x = fmaf(-x.y, y.y, s.x);
        s.y = fmaf(x.x, y.y, s.y);
        s.y = fmaf(x.y, y.x, s.y);
      }
      acc[q] = s;
      big = fmaxf(big, fmaxf(fabsf(s.x), fabsf(s.y)));
    }
    atomicMax(&s_max[k], __float_as_int(big));
    __syncthreads();
    q = 0;
    for (int e = threadIdx.x; e < n * n; e += blockDim.x, ++q) R[e] = acc[q];
    __syncthreads();
  }
  if (threadIdx.x < kExpStride) {
    const int k = threadIdx.x;
    int ek = 0;
    if (k == 1) ek = e1;
    if (k >= 2 && k <= top) {
      const int f = (s_max[k] >> 23) & 255;
      if (f < 20 || f > 250) s_bad = 1;  // zero, vanishing or not finite
      ek = k * e1 + f - 126 + kFxRoom;
    }
    P.exps[(int64_t)b * kExpStride + k] = ek;
  }
  __syncthreads();
  if (threadIdx.x == 0 && !s_bad) P.ok[b] = 1;
}

// Pair sums (see pair_terms_elems) of kSumBlocks blocks of one matrix: Q_p of
// each entry by two fixed-point products, then the sums over the subsets of
// the low and of the high pairs.
__global__ void __launch_bounds__(256) terms_sums_kernel(const TermsLaunch P) {
  __shared__ int4 Q[kSumBlocks * 4 * kMaxH];
  dependency_wait();
  const int hm = P.stage_h, chunks = (hm * (hm + 1) / 2 + kSumBlocks - 1) / kSumBlocks;
  const int b = blockIdx.x / chunks, b0 = (blockIdx.x - b * chunks) * kSumBlocks;
  const int n = P.pats[b].n, h = n >> 1, nb = h * (h + 1) / 2;
  if (n < 6 || (n & 1) || b0 >= nb || P.sum_off[b] < 0 || P.ok[b] == 0) return;  // uniform
  const int* ex = P.exps + (int64_t)b * kExpStride;
  const int sh = 27 + ex[2] - 2 * ex[1];
  if (!fx_shift_ok(sh)) {
    if (threadIdx.x == 0) P.ok[b] = 0;
    return;
  }
  const int4* mat = P.mat + P.mat_off[b];
  const int cnt = min(kSumBlocks, nb - b0);
  bool over = false;
  auto entry = [&](int i, int j) -> int4 {  // A(i, j)
    const int r = i >> 1, c = j >> 1;
    const int el = (r <= c) ? 2 * (i & 1) + (j & 1) : 2 * (j & 1) + (i & 1);
    return __ldg(mat + 4 * blk_index(r, c, h) + el);
  };
  for (int t = threadIdx.x; t < cnt * 4 * h; t += blockDim.x) {
    const int p = t % h, el = (t / h) & 3, k = b0 + t / (4 * h);
    int r, c;
    if (k >= h * (h - 1) / 2) {
      r = c = k - h * (h - 1) / 2;
    } else {
      c = 1;
      while (c * (c + 1) / 2 <= k) ++c;
      r = k - c * (c - 1) / 2;
    }
    const int i = 2 * r + (el >> 1), j = 2 * c + (el & 1);
    Fx q = fx_zero();
    const FxOp a0 = fx_load(entry(i, 2 * p)), a1 = fx_load(entry(i, 2 * p + 1));
    fx_mac(q, a0, -a0.hi, fx_load(entry(2 * p + 1, j)));
    fx_mac(q, a1, -a1.hi, fx_load(entry(2 * p, j)));
    Q[t] = fx_entry(q, sh, over);
  }
  __syncthreads();
  const int hl = pair_split_lo(h), W = pair_sums_width(h);
  int4* out = P.mat + P.sum_off[b] + (int64_t)b0 * W * 4;
  for (int t = threadIdx.x; t < cnt * W * 4; t += blockDim.x) {
    const int el = t & 3, w = (t >> 2) % W, k = (t >> 2) / W;
    const bool low = w < (1 << hl);
    unsigned m = low ? (unsigned)w : (unsigned)(w - (1 << hl)) << hl;
    int hr = 0, hi = 0;
    float lr = 0.0f, li = 0.0f;
    for (; m; m &= m - 1) {
      const int4 v = Q[(k * 4 + el) * h + __ffs(m) - 1];
      hr += v.x;
      hi += v.y;
      lr += __int_as_float(v.z);
      li += __int_as_float(v.w);
    }
    const int2 x = fx_pack(hr, lr, over), y = fx_pack(hi, li, over);
    out[t] = make_int4(x.x, y.x, x.y, y.y);
  }
  if (over) P.ok[b] = 0;
}

// R_c = R_a X R_b in 2 x 2 blocks: block (r, c) sums over the pairs t the
// products of block (r, t) of R_a with block (t, c) of R_b, rows swapped; per
// step eight 16-byte loads feed eight multiply-adds. A block
// below the diagonal is its mirror with elements 1 and 2 exchanged. Lanes take
// consecutive blocks (one column, consecutive rows): R_b's loads are then
// broadcasts and R_a's fall into different banks (their numbers step by 1 or
// run through the triangular numbers, which differ mod 8).
__device__ __forceinline__ void fx_prod(int4* __restrict__ dst, const int4* __restrict__ Ra,
                                        const int4* __restrict__ Rb, const unsigned short* __restrict__ rc, int s,
                                        int E, int sh, int l, int L, bool& over) {
  const int D = s * (s - 1) / 2;
  for (int e0 = 0; e0 < E; e0 += L) {
    const int e = min(e0 + l, E - 1);
    int r, c;
    if (e >= D) {
      r = c = e - D;
    } else {
      const int v = rc[e];
      r = v & 255;
      c = v >> 8;
    }
    Fx c00 = fx_zero(), c01 = c00, c10 = c00, c11 = c00;
    const int rr = r * (r - 1) / 2, cc = c * (c - 1) / 2;
    int tt = 0;  // t (t - 1) / 2
#pragma unroll 1
    for (int t = 0; t < s; ++t) {
      const int ia = (t > r) ? tt + r : (t == r) ? D + r : rr + t;
      const int ib = (t > c) ? tt + c : (t == c) ? D + c : cc + t;
      const int a1 = (t < r) ? 2 * E : E, b1 = (t > c) ? 2 * E : E;
      const int4* pa = Ra + ia;
      const int4* pb = Rb + ib;
      const FxOp y10 = fx_load(pb[3 * E - b1]), y00 = fx_load(pb[0]), y11 = fx_load(pb[3 * E]), y01 = fx_load(pb[b1]);
      {
        const FxOp x0 = fx_load(pa[0]), x1 = fx_load(pa[a1]);
        const int n0 = -x0.hi, n1 = -x1.hi;
        fx_mac(c00, x0, n0, y10);
        fx_mac(c01, x0, n0, y11);
        fx_mac(c00, x1, n1, y00);
        fx_mac(c01, x1, n1, y01);
      }
      {
        const FxOp x0 = fx_load(pa[3 * E - a1]), x1 = fx_load(pa[3 * E]);
        const int n0 = -x0.hi, n1 = -x1.hi;
        fx_mac(c10, x0, n0, y10);
        fx_mac(c11, x0, n0, y11);
        fx_mac(c10, x1, n1, y00);
        fx_mac(c11, x1, n1, y01);
      }
      tt += t;
    }
    if (e0 + l < E) {
      dst[e] = fx_entry(c00, sh, over);
      dst[E + e] = fx_entry(c01, sh, over);
      dst[2 * E + e] = fx_entry(c10, sh, over);
      dst[3 * E + e] = fx_entry(c11, sh, over);
    }
  }
}

// Traces, this lane's share, as 64-bit integers (tr X R_a X R_b: in
// 2^{E_a + E_b - 54}, tr X R_a: in 2^{E_a - 47}). Blocks above the diagonal stand for their
// mirrors too: they come first, and the sum is doubled before the diagonal
// ones; within a block the square's terms pair up as well.
__device__ __forceinline__ longlong2 fx_tr2(const int4* __restrict__ Ra, const int4* __restrict__ Rb, int s, int E,
                                            int l, int L) {
  const int D = s * (s - 1) / 2;
  const bool square = Ra == Rb;
  Fx c = fx_zero();
  bool twice = false;
  for (int e = l; e < E; e += L) {
    if (e >= D && !twice) {
      c.rh <<= 1;
      c.ih <<= 1;
      c.rm *= 2.0f;
      c.im *= 2.0f;
      twice = true;
    }
    const FxOp x00 = fx_load(Ra[e]), x01 = fx_load(Ra[E + e]);
    fx_mac(c, x00, -x00.hi, fx_load(Rb[3 * E + e]));
    fx_mac(c, x01, -x01.hi, fx_load(Rb[2 * E + e]));
    if (!square) {
      const FxOp x10 = fx_load(Ra[2 * E + e]), x11 = fx_load(Ra[3 * E + e]);
      fx_mac(c, x10, -x10.hi, fx_load(Rb[E + e]));
      fx_mac(c, x11, -x11.hi, fx_load(Rb[e]));
    }
  }
  longlong2 w;
  w.x = c.rh + __float2ll_rn(64.0f * c.rm);
  w.y = c.ih + __float2ll_rn(64.0f * c.im);
  const int up = (twice ? 0 : 1) + (square ? 1 : 0);
  w.x <<= up;
  w.y <<= up;
  return w;
}
__device__ __forceinline__ longlong2 fx_tr1(const int4* __restrict__ Ra, int s, int E, int l, int L) {
  longlong2 w = make_longlong2(0, 0);
  for (int r = l; r < s; r += L) {
    const int4 v = Ra[E + s * (s - 1) / 2 + r];
    w.x += ((long long)v.x << 20) + __float2int_rn(__int_as_float(v.z) * 0x1p20f);
    w.y += ((long long)v.y << 20) + __float2int_rn(__int_as_float(v.w) * 0x1p20f);
  }
  w.x <<= 1;
  w.y <<= 1;
  return w;
}

// Persistent warps over work items (as haf_subsets_kernel): a warp takes
// 32 / L subsets of one size at a time, L lanes each. Six to ten warps an SM
// (shared memory sets the number) leave latency in sight, so loads are issued
// ahead of their use and sums run two at a time. 4096 patterns of n = 16: this
// kernel 2.66 -> 2.35 ms (with one load in flight, each trace summed alone);
// with every part timed by leaving it out, products take 1.1 ms of it, their
// rounding a third of that, traces and loads 0.6, the series 0.3, the sums over
// lanes 0.3 (before the pairing). 80 patterns of n = 28 and 30: products 22 of
// 40 ms, at six warps an SM.
__global__ void __launch_bounds__(kTermsWarps * 32, 1) haf_terms_kernel(const TermsLaunch P) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ Tables tab;
  __shared__ unsigned short rc[kMaxH * (kMaxH - 1) / 2];
  if (threadIdx.x <= kMaxH) {
    const int a = threadIdx.x;
    int c = 1;
    for (int b = 0; b <= kMaxH; ++b) {  // C(a, b) = C(a, b-1) (a-b+1) / b
      tab.binom[a][b] = (b <= a) ? c : 0;
      if (b < a) c = c * (a - b) / (b + 1);
    }
    tab.inv2k[a] = (a == 0) ? 0.0 : 1.0 / (2.0 * a);
    for (int r = 0; r < a && a < kMaxH; ++r) rc[a * (a - 1) / 2 + r] = (unsigned short)(r | (a << 8));
  }
  dependency_wait();
  __syncthreads();
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char* wbase = smem + (size_t)warp * P.warp_bytes;
  double* sc = reinterpret_cast<double*>(wbase);      // trace k's unit, k = 1..16 at k - 1
  double* cn = sc + kMaxH;                            // bound on its rounding over 2k
  int* ex = reinterpret_cast<int*>(cn + kMaxH);       // E_k
  longlong2* stage = reinterpret_cast<longlong2*>(wbase + kTermsHeader);
  const int sts = stage_stride(P.stage_h), slots = stage_slots(P.stage_h);
  unsigned char* gbase = wbase + kTermsHeader + terms_stage_bytes(P.stage_h);

  for (;;) {
    int it = 0;
    if (lane == 0) it = atomicAdd(P.counter, 1);
    it = __shfl_sync(FULL, it, 0);
    if (it >= P.n_items) break;
    const WorkItem w = P.items[it];
    if ((P.skip != nullptr && P.skip[w.pat] != 0) || P.ok[w.pat] == 0) {
      if (lane == 0) P.kparts[w.part] = make_double2(0.0, 0.0);
      continue;
    }
    const int n = P.pats[w.pat].n, h = n >> 1;
    const bool whole = w.s_last > w.s;
    const int s_first = w.s, s_last = whole ? w.s_last : w.s;
    const int4* mat = P.mat + P.mat_off[w.pat];
    const int64_t so = P.sum_off[w.pat];
    const int4* sums = (so >= 0) ? P.mat + so : nullptr;
    const int hl = pair_split_lo(h), W = pair_sums_width(h);
    bool over = false;
    __syncwarp();
    if (lane < kExpStride) ex[lane] = P.exps[(int64_t)w.pat * kExpStride + lane];
    __syncwarp();
    // units and rounding bounds of the traces, by the schedule's ops (the
    // power each buffer holds in pw, four bits a buffer)
    {
      unsigned pw = 1;
      for (int o = 0; o < kMaxOps; ++o) {
        const SchedOp op = c_sched[h][o];
        if (op.kind == kEnd) break;
        const int ka = (pw >> (4 * op.a)) & 15, kb = (pw >> (4 * op.b)) & 15;
        if (op.kind == kProd) {
          pw = (pw & ~(15u << (4 * op.k))) | (unsigned)(ka + kb) << (4 * op.k);
          if (!fx_shift_ok(27 + ex[ka + kb] - ex[ka] - ex[kb])) over = true;
        } else if (lane == 0) {
          const int u = (op.kind == kTr1) ? ex[ka] - 47 : ex[ka] + ex[kb] - 54;
          if (u < -1000 || u > 1000) over = true;
          sc[op.k - 1] = __hiloint2double((max(min(u, 1000), -1000) + 1023) << 20, 0);
          // n entries off by 2^-49 of their range, against the other factor's largest
          cn[op.k - 1] = (double)n * sc[op.k - 1] * ((op.kind == kTr1) ? 0.25 : 8.0) * tab.inv2k[op.k];
        }
      }
      over = __any_sync(FULL, over);
      __syncwarp();
    }
    if (over) {
      if (lane == 0) {
        P.ok[w.pat] = 0;
        P.kparts[w.part] = make_double2(0.0, 0.0);
      }
      continue;
    }
    double kap = 0.0, noise = 0.0;
    int staged = 0;

    // the exponential series (as in haf_subsets_kernel) of one staged subset
    // per lane; d f / d tr_k = e_{h-k} / (2k) carries the traces' rounding
    auto flush = [&]() {
      if (lane < staged) {
        double2 e[kMaxH];
        longlong2* raw = stage + lane * sts;
        double2* pq = reinterpret_cast<double2*>(raw);
#pragma unroll 1
        for (int k = 0; k < h; ++k) {
          const longlong2 v = raw[k];
          pq[k] = make_double2((double)v.x * sc[k], (double)v.y * sc[k]);
        }
        double2 f = mk<double>(1.0, 0.0);
        double nz = cn[h - 1];
#pragma unroll 1
        for (int k = 1; k <= h; ++k) {
          double2 a = pq[k - 1];
#pragma unroll 1
          for (int j = 1; j < k; ++j) a = cfma<double>(pq[j - 1], e[k - j], a);
          const double c = tab.inv2k[k];
          f = mk<double>(a.x * c, a.y * c);
          if (k < h) {
            e[k] = f;
            nz = fma(cn[h - k - 1], fabs(f.x) + fabs(f.y), nz);
          }
        }
        kap += fabs(f.x) + fabs(f.y);
        noise += nz;
      }
      staged = 0;
      __syncwarp();
    };

    for (int s = s_first; s <= s_last; ++s) {
      const int E = s * (s + 1) / 2, D = s * (s - 1) / 2;
      const int L = terms_lanes(s, h, P.warp_bytes, P.stage_h);
      const int G = 32 / L, g = lane / L, l = lane - g * L;
      int4* buf = reinterpret_cast<int4*>(gbase + (size_t)g * terms_group_bytes(s, h, L));
      int* pairs = reinterpret_cast<int*>(buf + sched_nbuf(h) * 4 * E);
      const int count = whole ? tab.binom[h][s] : w.count, rank0 = whole ? 0 : w.rank0;
      const int rounds = (count + G - 1) / G;
      unsigned gmask = 0;
      for (int rd = 0; rd < rounds; ++rd) {
        if (staged + G > slots) flush();
        const int js = g * rounds + rd;
        const bool active = js < count;
        if (rd == 0) {
          int r = rank0 + (active ? js : 0), c = h - 1;
          for (int i = s; i >= 1; --i) {
            while (tab.binom[c][i] > r) --c;
            r -= tab.binom[c][i];
            gmask |= 1u << c;
            --c;
          }
        } else if (active) {  // the next larger mask with s bits
          const unsigned u = gmask & (0u - gmask), v = gmask + u;
          gmask = v + (((v ^ gmask) >> 2) >> (__ffs(u) - 1));
        }
        {
          unsigned m = gmask;
          for (int t = 0; t < s; ++t) {
            if ((t & (L - 1)) == l) pairs[t] = __ffs(m) - 1;
            m &= m - 1;
          }
        }
        __syncwarp();
        // R_1 (and R_2 from the pair sums): the subset's blocks
        const bool have2 = sums != nullptr && h >= 3;
        const int klo = (int)(gmask & ((1u << hl) - 1)), khi = (1 << hl) + (int)(gmask >> hl);
        // (the loads of four entries are issued before the first is used)
        for (int f0 = l; f0 < 4 * E; f0 += 4 * L) {
          int4 v[4], x[4], y[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int f = f0 + u * L, e = f >> 2, el = f & 3;
            if (f < 4 * E) {
              int r, c;
              if (e >= D) {
                r = c = e - D;
              } else {
                const int z = rc[e];
                r = z & 255;
                c = z >> 8;
              }
              const int src = blk_index(pairs[r], pairs[c], h);
              v[u] = __ldg(mat + 4 * src + el);
              if (have2) {
                const int4* q = sums + ((int64_t)src * W) * 4 + el;
                x[u] = __ldg(q + 4 * klo);
                y[u] = __ldg(q + 4 * khi);
              }
            }
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int f = f0 + u * L, e = f >> 2, el = f & 3;
            if (f < 4 * E) {
              buf[el * E + e] = v[u];
              if (have2) {
                const int2 re = fx_pack(x[u].x + y[u].x, __int_as_float(x[u].z) + __int_as_float(y[u].z), over);
                const int2 im = fx_pack(x[u].y + y[u].y, __int_as_float(x[u].w) + __int_as_float(y[u].w), over);
                buf[4 * E + el * E + e] = make_int4(re.x, im.x, re.y, im.y);
              }
            }
          }
        }
        __syncwarp();
        longlong2* const row = stage + (staged + g) * sts;
        unsigned pw = 1;
        longlong2 wait = make_longlong2(0, 0);
        int wait_k = 0;  // 0: none waiting
        for (int o = 0; o < kMaxOps; ++o) {
          const SchedOp op = c_sched[h][o];
          if (op.kind == kEnd) break;
          const int ka = (pw >> (4 * op.a)) & 15, kb = (pw >> (4 * op.b)) & 15;
          const int4* Ra = buf + op.a * 4 * E;
          const int4* Rb = buf + op.b * 4 * E;
          if (op.kind == kProd) {
            if (!(have2 && ka + kb == 2))
              fx_prod(buf + op.k * 4 * E, Ra, Rb, rc, s, E, 27 + ex[ka + kb] - ex[ka] - ex[kb], l, L, over);
            pw = (pw & ~(15u << (4 * op.k))) | (unsigned)(ka + kb) << (4 * op.k);
          } else {
            // the lanes' shares are summed two traces at a time, as group_sum2
            // does (half the lanes carry one, half the other); they are whole
            // numbers, so the order does not matter
            const longlong2 t = (op.kind == kTr1) ? fx_tr1(Ra, s, E, l, L) : fx_tr2(Ra, Rb, s, E, l, L);
            if (L == 1) {
              row[op.k - 1] = active ? t : make_longlong2(0, 0);
            } else if (wait_k == 0) {
              wait = t;
              wait_k = op.k;
            } else {
              const int half = L >> 1;
              const bool up = (l & half) != 0;
              const longlong2 out = up ? wait : t;
              longlong2 keep = up ? t : wait;
              keep.x += __shfl_xor_sync(FULL, out.x, half);
              keep.y += __shfl_xor_sync(FULL, out.y, half);
              for (int off = half >> 1; off > 0; off >>= 1) {
                keep.x += __shfl_xor_sync(FULL, keep.x, off);
                keep.y += __shfl_xor_sync(FULL, keep.y, off);
              }
              if ((l & (half - 1)) == 0) row[(up ? op.k : wait_k) - 1] = active ? keep : make_longlong2(0, 0);
              wait_k = 0;
            }
          }
          __syncwarp();
        }
        if (wait_k != 0) {  // uniform over the warp
          for (int off = L >> 1; off > 0; off >>= 1) {
            wait.x += __shfl_xor_sync(FULL, wait.x, off);
            wait.y += __shfl_xor_sync(FULL, wait.y, off);
          }
          if (l == 0) row[wait_k - 1] = active ? wait : make_longlong2(0, 0);
          __syncwarp();
        }
        staged += G;
        if (staged == slots || (rd == rounds - 1 && s == s_last)) flush();
      }
    }
    for (int off = 16; off > 0; off >>= 1) {
      kap += __shfl_xor_sync(FULL, kap, off);
      noise += __shfl_xor_sync(FULL, noise, off);
    }
    if (__any_sync(FULL, over) && lane == 0) P.ok[w.pat] = 0;
    if (lane == 0) P.kparts[w.part] = make_double2(kap, noise);
  }
}

// One warp per matrix: the sum over its items; a matrix that left the range,
// or whose rounding bound is above 2^-33 of the sum, goes to the FP64 kernel,
// whose item count the last block sets (0 where no matrix does).
__global__ void __launch_bounds__(256) terms_check_kernel(const TermsLaunch P) {
  dependency_wait();
  const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  bool redo = false;
  for (int b = blockIdx.x * wpb + (threadIdx.x >> 5); b < P.batch; b += gridDim.x * wpb) {
    const PatDesc d = P.pats[b];
    const bool mine = d.n >= 2 && !(d.n & 1) && !(P.skip != nullptr && P.skip[b] != 0);
    double K = 0.0, noise = 0.0;
    bool fine = true;
    if (mine) {
      for (int q = d.item_begin + lane; q < d.item_end; q += 32) {
        const double2 v = P.kparts[q];
        K += v.x;
        noise += v.y;
      }
      int span = 1;
      while (span < min(32, d.item_end - d.item_begin)) span <<= 1;
      for (int off = span >> 1; off > 0; off >>= 1) {
        K += __shfl_xor_sync(0xffffffffu, K, off);
        noise += __shfl_xor_sync(0xffffffffu, noise, off);
      }
      if (lane == 0) fine = P.ok[b] != 0 && noise <= 0x1p-33 * K && K < INFINITY;
    }
    if (lane == 0) {
      P.ksum[b] = K;
      P.ok[b] = fine ? 1 : 0;
      redo |= !fine;
    }
  }
  if (redo) atomicAdd(P.n_redo, 1);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0 && atomicAdd(P.blocks_done, 1u) == gridDim.x - 1) {
    __threadfence();
    *P.fp64_items = __ldcg(P.n_redo) ? P.n_items : 0;
  }
}
