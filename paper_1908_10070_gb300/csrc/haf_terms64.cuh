// The same moduli in FP64 (included by haf_subsets.cu after haf_terms.cuh):
// for the orders below kTermsFixedMin, and for the matrices that the
// fixed-point kernels could not do or gave back.
//
// Below order 12 kappa from the fixed-point sum is off by more than kappa from
// the subset sum was, whose Hafnian brings the larger part of its error (60
// matrices of four kinds an order, Haar and random; largest, subset sum / fixed
// point / now: n = 4 2.0e-15 / 1.2e-14 / 4e-16, n = 8 1.2e-14 / 2.2e-14 / 2e-15,
// n = 10 2.4e-14 / 3.6e-14 / 3e-15). From 12 on it is off by less, in the mean,
// the root mean square and the largest of each kind (n = 12 at most 7.2e-15,
// 2.1e-14, 1.5e-13 / 3.5e-15, 4.5e-15, 1.4e-14; largest at n = 16 9.3e-13 /
// 1.1e-14, at 24 1.2e-11 / 1.1e-14), and FP64 would take twice the time (1024
// of n = 12 318 us instead of 165, 399 by the subset sum). Here sum |f| is
// within 1e-15 of its value, as the powers gave it.
//
// The same Krylov vectors and series as there (a third of the products of the
// powers of a subset's matrix at order 16, a quarter at 30), on the matrix
// scaled to entries below 1 by a power of two (exact). Bound by the FP64 pipe,
// so the layout only has to keep its lanes filled: rows as lanes, then a
// subset's series per lane. Two launches whatever the order: a block takes 128
// neighbouring masks and recomputes the series of the prefixes they share (a
// quarter of the Krylov products at order 30) instead of a launch per level.
// As many blocks as are resident stride over the items of either, and leave at
// once when no matrix is left to them (the usual case).

constexpr int kCoefs64 = (kMatchMaxN / 2 + 5) / 6;  // most coefficients per lane (6 lanes a subset at least)
constexpr int kSeries64 = 128;                      // threads (columns) of a block of the series kernel

// FP64 terms of matrix b: not the repeated-row sum's, not done in fixed point.
__device__ __forceinline__ bool terms64_wanted(const TermsLaunch& P, int b) {
  return P.ok[b] == 0 && (P.skip == nullptr || P.skip[b] == 0);
}
__device__ __forceinline__ void zmac(double2& c, double2 a, double2 b) {
  c.x = fma(a.x, b.x, c.x);
  c.x = fma(-a.y, b.y, c.x);
  c.y = fma(a.x, b.y, c.y);
  c.y = fma(a.y, b.x, c.y);
}

// D_S of every subset of a small order, D_S^{-1/2} of every one of a larger (in
// the place of the fixed-point path's D). Item: a part of a matrix, as a block
// of terms_delta_kernel. The root is taken by the subset's lanes for the larger
// orders, an eighth more work than by one thread of the series kernel, whose
// chain was twice as long for it (a lone matrix of order 24: 635 -> 500 us);
// small orders come in numbers and have short chains (4096 of order 8 took 245
// us with the root here, 207 there).
__global__ void __launch_bounds__(kDeltaThreads) terms64_delta_kernel(const TermsLaunch P, const TermsChunk C) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int binom[kMaxH + 1][kMaxH + 1], rows[kMaxN], s_max;
  __shared__ double inv[kMaxH + 1];  // -1 / k
  if (threadIdx.x >= 1 && threadIdx.x <= kMaxH) inv[threadIdx.x] = -1.0 / threadIdx.x;
  if (threadIdx.x <= kMaxH) {
    const int a = threadIdx.x;
    int c = 1;
    for (int b = 0; b <= kMaxH; ++b) {
      binom[a][b] = (b <= a) ? c : 0;
      if (b < a) c = c * (a - b) / (b + 1);
    }
  }
  dependency_wait();
  __syncthreads();
  const int items = C.small64 < C.items64 && *P.left ? C.items64 : C.small64;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int item = blockIdx.x; item < items; item += gridDim.x) {
    int g = C.n_groups - 1;  // (items are numbered from the smallest order on)
    while (g > 0 && item >= C.g[g - 1].item64) --g;
    const TermsGroup& G = C.g[g];
    const int n = G.n, h = n >> 1, q = (item - G.item64) / G.parts64, part = (item - G.item64) - q * G.parts64;
    const int b = P.order[G.first + q];
    if (!terms64_wanted(P, b)) continue;  // uniform
    const bool small = n < kTermsFixedMin;
    const PatDesc d = P.pats[b];
    double2* root = reinterpret_cast<double2*>(C.scratch) + G.off + (int64_t)q * G.stride + n * n;
    double2* M = reinterpret_cast<double2*>(smem);
    const int ld = n + 1;
    if ((int)threadIdx.x < n) {
      int pos = default_pos(threadIdx.x, h);
      if (P.perm != nullptr && P.perm_off[b] >= 0) pos = P.perm[P.perm_off[b] + threadIdx.x];
      int v = (d.idx_off >= 0) ? P.idx[d.idx_off + pos] : pos;
      if (P.m_bound > 0 && (v < 0 || v >= P.m_bound)) {
        P.status[b] = 1;
        v = 0;
      }
      rows[threadIdx.x] = v;
    }
    if (threadIdx.x == 0) s_max = 0;
    __syncthreads();
    const double2* src2 = reinterpret_cast<const double2*>(P.src) + d.src_off;
    int mine = 0;
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
      const int r = e / n, c = e - r * n;
      double2 v = make_double2(0.0, 0.0);
      if (r != c) v = __ldg(src2 + (int64_t)rows[min(r, c)] * d.ld + rows[max(r, c)]);
      M[r * ld + c] = v;
      mine = max(mine, max((__double2hiint(v.x) >> 20) & 2047, (__double2hiint(v.y) >> 20) & 2047));
    }
    mine = __reduce_max_sync(0xffffffffu, mine);
    if (lane == 0) atomicMax(&s_max, mine);
    __syncthreads();
    // every |entry| < 2^e1 (entries that are not finite stay so)
    const int e1 = min(max(s_max - 1022, -1000), 1000);
    const double unit = __hiloint2double((1023 - e1) << 20, 0);
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
      double2& v = M[(e / n) * ld + e % n];
      v.x *= unit;
      v.y *= unit;
    }
    if (part == 0 && threadIdx.x == 0) P.exps[(int64_t)b * kExpStride] = e1;
    __syncthreads();
    const int steps = (h - 1) / 2;  // vectors u_0 .. u_steps
    unsigned char* wbase = smem + (size_t)n * ld * 16 + (size_t)warp * G.region;
    int s = 1, done = 0;  // rounds of the sizes below s
    for (int r = part * nw + warp;; r += G.parts64 * nw) {
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
      double2* V = reinterpret_cast<double2*>(wbase + (size_t)gi * terms_group_bytes(s, h));
      const int sp = s - 1, N = 2 * sp;
      double2* mom = V + (steps + 1) * 2 * N;  // a, b, c at 3 (k - 1) + 0, 1, 2
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
      const bool row_mine = l < N;
      const double2* row = M + (row_mine ? 2 * pairs[l >> 1] + (l & 1) : 0) * ld;
      if (row_mine) {
        V[l] = row[2 * p];
        V[N + l] = row[2 * p + 1];
      }
      __syncwarp();
      for (int k = 1; k <= steps; ++k) {
        if (row_mine) {
          const double2* U = V + (k - 1) * 2 * N;
          double2 ca = make_double2(0.0, 0.0), cb = ca, cc = ca, cd = ca;
#pragma unroll 1
          for (int t = 0; t < sp; ++t) {
            const int c = 2 * pairs[t];
            const double2 x0 = row[c], x1 = row[c + 1];
            zmac(ca, x0, U[2 * t + 1]);
            zmac(cb, x0, U[N + 2 * t + 1]);
            zmac(cc, x1, U[2 * t]);
            zmac(cd, x1, U[N + 2 * t]);
          }
          V[k * 2 * N + l] = make_double2(ca.x + cc.x, ca.y + cc.y);
          V[k * 2 * N + N + l] = make_double2(cb.x + cd.x, cb.y + cd.y);
        }
        __syncwarp();
      }
      // the walks' sums, one a lane; the three of x^1, which cost nothing, last
      for (int r1 = l; l < L && r1 < 3 * h; r1 += L) {
        const int t = 3 * h - 1 - r1, k = t / 3 + 1, type = t - 3 * (k - 1);
        double2 v = make_double2(0.0, 0.0);
        if (k == 1) {
          if (type == 1) v = M[2 * p * ld + 2 * p + 1];
        } else {
          const int i = (k - 2) >> 1, j = k - 2 - i;
          const double2* x = V + i * 2 * N + (type == 2 ? N : 0);
          const double2* y = V + j * 2 * N + (type == 0 ? 0 : N);
          double2 w = make_double2(0.0, 0.0);
          for (int r2 = 0; r2 < N; r2 += 2) {
            zmac(v, x[r2], y[r2 + 1]);
            zmac(w, x[r2 + 1], y[r2]);
          }
          v.x += w.x;
          v.y += w.y;
        }
        mom[t] = v;
      }
      __syncwarp();
      // coefficient k = h - l - m L of D_S = 1 - 2 b + b^2 - a c
      double2 acc[kCoefs64];
#pragma unroll
      for (int m = 0; m < kCoefs64; ++m) {
        const int k = h - l - m * L;
        if (l >= L || k < 1) continue;
        const double2 bk = mom[3 * (k - 1) + 1];
        double2 c = make_double2(-2.0 * bk.x, -2.0 * bk.y);
        for (int i = 1; i < k; ++i) {
          const double2 ai = mom[3 * (i - 1)];
          zmac(c, make_double2(-ai.x, -ai.y), mom[3 * (k - i - 1) + 2]);
          if (2 * i <= k) {
            const double2 bi = mom[3 * (i - 1) + 1];
            const double f = 2 * i == k ? 1.0 : 2.0;  // b_i b_(k-i) twice
            zmac(c, make_double2(bi.x * f, bi.y * f), mom[3 * (k - i - 1) + 1]);
          }
        }
        acc[m] = c;
      }
      __syncwarp();  // the walks' sums are read: D_S and its root take their place
      double2 *ds = mom, *ys = mom + h;
#pragma unroll
      for (int m = 0; m < kCoefs64; ++m) {
        const int k = h - l - m * L;
        if (l >= L || k < 1) continue;
        ds[k - 1] = acc[m];
        acc[m].x *= 0.5 * k;
        acc[m].y *= 0.5 * k;
      }
      if (small) {
        __syncwarp();
        for (int k = l; active && k < h; k += L) root[(int64_t)mask * h + k] = ds[k];
      }
      // y = D_S^{-1/2}: -k y_k = sum_i (k - i / 2) d_i y_{k-i}, each y_j added to
      // the later sums as it is found
      for (int j = small ? h + 1 : 1; j <= h; ++j) {
#pragma unroll
        for (int m = 0; m < kCoefs64; ++m)
          if (l < L && h - l - m * L == j) {
            const double2 y = make_double2(acc[m].x * inv[j], acc[m].y * inv[j]);
            ys[j - 1] = y;
            if (active) root[(int64_t)mask * h + j - 1] = y;
          }
        __syncwarp();
        const double2 y = ys[j - 1];
#pragma unroll
        for (int m = 0; m < kCoefs64; ++m) {
          const int k = h - l - m * L;
          if (l >= L || k <= j) continue;
          const double f = 0.5 * (k + j);
          const double2 d2 = ds[k - j - 1];
          zmac(acc[m], make_double2(d2.x * f, d2.y * f), y);
        }
      }
      __syncwarp();
    }
    __syncthreads();  // before the next item's matrix
  }
}

// The series and sum |f|_1. Item: 128 columns, one a thread: the masks of 128 /
// 2^h matrices for h <= 7, else the masks with one choice J of the pairs from 7
// on of one matrix; its blocks' sums meet in order in the block that ends last.
// (With 256 columns, two warps an SM quarter, a lone matrix took twice as long.)
__global__ void __launch_bounds__(kSeries64) terms64_series_kernel(const TermsLaunch P, const TermsChunk C) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double red[kSeries64], inv[kMaxH + 1];  // -1 / k
  __shared__ int s_last;
  if (threadIdx.x >= 1 && threadIdx.x <= kMaxH) inv[threadIdx.x] = -1.0 / threadIdx.x;
  constexpr int ld = kSeries64 + 1, bits = 7;
  dependency_wait();
  __syncthreads();
  const bool left = C.small64 < C.items64 && *P.left != 0;
  const int col = threadIdx.x;
  // coefficient k of a column at [k - 1][column]: D_S^{-1/2}, and G_S
  double2* ys = reinterpret_cast<double2*>(smem);
  double2* gs = ys + C.hmax64 * ld;
  int first = 0;  // items of the groups before
  for (int g = 0; g < C.n_groups; ++g) {
    const TermsGroup& G = C.g[g];
    const int n = G.n, h = n >> 1, hl = min(h, bits), per = kSeries64 >> hl;
    const int items = (n < kTermsFixedMin || left) ? (h <= bits ? (G.count + per - 1) / per : G.count << (h - bits)) : 0;
    int item = (blockIdx.x + gridDim.x - first % gridDim.x) % gridDim.x;  // goes on where the group before ended
    first += items;
    for (; item < items; item += gridDim.x) {
      const int low = col & ((1 << hl) - 1);
      const int q = h <= bits ? item * per + (col >> hl) : item >> (h - bits);
      const int J = h <= bits ? 0 : item & ((1 << (h - bits)) - 1);
      const int b = q < G.count ? P.order[G.first + q] : -1;
      const bool mine = b >= 0 && terms64_wanted(P, b);
      if (!__syncthreads_or(mine)) continue;  // (also: the item before is done with the shared arrays)
      double2* base = reinterpret_cast<double2*>(C.scratch) + G.off + (int64_t)q * G.stride;
      // the delta kernel's series of a mask into the thread's column
      auto load = [&](int S) {
        const double2* y = base + n * n + (int64_t)S * h;
#pragma unroll 4
        for (int k = 0; k < h; ++k) ys[k * ld + col] = y[k];
      };
      // coefficient k of G_S' y (constant terms 1)
      auto product = [&](int k, const double2* gp, const double2* y) {
        const double2 t = gp[(k - 1) * ld], u = y[(k - 1) * ld];
        double2 c = make_double2(t.x + u.x, t.y + u.y), e = make_double2(0.0, 0.0);
        int i = 1;
        for (; i + 1 < k; i += 2) {
          zmac(c, gp[(i - 1) * ld], y[(k - i - 1) * ld]);
          zmac(e, gp[i * ld], y[(k - i - 2) * ld]);
        }
        if (i < k) zmac(c, gp[(i - 1) * ld], y[(k - i - 1) * ld]);
        return make_double2(c.x + e.x, c.y + e.y);
      };
      if (mine && low != 0) {
        load(low);
        if (n < kTermsFixedMin) {  // D_S so far: -k y_k = sum_i (k - i / 2) d_i y_{k-i}, y_0 = 1
          for (int k = 1; k <= h; ++k) gs[(k - 1) * ld + col] = ys[(k - 1) * ld + col];
          for (int k = 1; k <= h; ++k) {
            const double2 d = gs[(k - 1) * ld + col];
            double2 c = make_double2(0.5 * k * d.x, 0.5 * k * d.y);
            for (int i = 1; i < k; ++i) {
              const double f = k - 0.5 * i;
              const double2 di = gs[(i - 1) * ld + col];
              zmac(c, make_double2(di.x * f, di.y * f), ys[(k - i - 1) * ld + col]);
            }
            ys[(k - 1) * ld + col] = make_double2(c.x * inv[k], c.y * inv[k]);
          }
        }
      } else {  // the empty set: G = 1
        for (int k = 0; k < h; ++k) ys[k * ld + col] = gs[k * ld + col] = make_double2(0.0, 0.0);
      }
      for (int p = 0; p < hl; ++p) {
        __syncthreads();
        for (int t = col; t < (per * h) << p; t += kSeries64) {
          const int c = t & ((per << p) - 1), k = h - t / (per << p);
          const int S = ((c >> p) << hl) + (1 << p) + (c & ((1 << p) - 1));  // the column of matrix c >> p
          gs[(k - 1) * ld + S] = product(k, gs + (S ^ (1 << p)), ys + S);
        }
      }
      __syncthreads();
      double2 f = gs[(h - 1) * ld + col];
      for (int rest = J, pre = 0; rest && mine; rest &= rest - 1) {  // (the thread's column alone)
        pre |= rest & -rest;
        load((pre << bits) | low);
        if (rest & (rest - 1)) {
          for (int k = h; k >= 1; --k) gs[(k - 1) * ld + col] = product(k, gs + col, ys + col);
        } else {
          f = product(h, gs + col, ys + col);
        }
      }
      red[col] = mine && (low != 0 || J != 0) ? fabs(f.x) + fabs(f.y) : 0.0;
      __syncthreads();
      for (int o = (1 << hl) >> 1; o > 0; o >>= 1) {
        if (low < o) red[col] += red[col + o];
        __syncthreads();
      }
      const int unit = mine ? h * P.exps[(int64_t)b * kExpStride] : 0;
      if (h <= bits) {
        if (mine && low == 0) P.ksum[b] = ldexp(red[col], unit);
        continue;
      }
      // one matrix: this block's share, and all shares in the block that ends last
      const int shares = 1 << (h - bits);
      double* parts = reinterpret_cast<double*>(base + n * n + ((int64_t)h << h));
      if (col == 0) {
        parts[J] = red[0];
        __threadfence();
        s_last = atomicAdd(P.done + b, 1) == shares - 1;
      }
      __syncthreads();
      if (!s_last) continue;
      __threadfence();
      double sum = 0.0;
      for (int i = col; i < shares; i += kSeries64) sum += __ldcg(parts + i);
      red[col] = sum;
      __syncthreads();
      for (int o = kSeries64 / 2; o > 0; o >>= 1) {
        if (col < o) red[col] += red[col + o];
        __syncthreads();
      }
      if (col == 0) P.ksum[b] = ldexp(red[0], unit);
    }
  }
}
