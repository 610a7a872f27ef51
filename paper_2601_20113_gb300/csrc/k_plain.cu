// Plain FP64 compression path: one CTA per block.
//
// Per block (Algorithm 1 step 3 of arXiv 2601.20113, with the readings of the
// pointwise-bound form):
//   Gram G = A^T A (cross-product SVD, Sec. 2.7.1)      FP64, sequential fma per entry
//   Jacobi eigensolve, round-robin ordering (Sec. 2.3)   FP64, the whole CTA, an entry a thread
//   projection C = A Vst (Sec. 2.5, Eq. 5)               FP64 fma chain per coefficient
//   quantization q = rint(C / delta)
//   bisection for the smallest rank with E(r) <= eps_l^2 (Sec. 2.4 Eq. 4, Eq. 6)
//   pointwise correction k = rint((x - xhat) / 2eb), escapes
//   per-block record size (raw if not smaller)
// Every floating-point operation that decides a stored value is written with
// an explicit rounding intrinsic, in the same order as the definitions, so the
// result is bit-identical to any IEEE implementation of those definitions.
//
// The FP64 pipe (about two lanes a clock and SM, 1/64 of the FP32 rate) bounds
// this form, so it is kept for the values that are FP64 by definition: the
// Gram chains, the eigensolve, and float64 fields' projection and decode.
// Elsewhere a decision that FP32 (float32 fields) or a product with a
// reciprocal (float64) settles beyond its own error bound is taken there, and
// the FP64 definition runs only where the bound leaves it open; conversions,
// finite tests and magnitude comparisons are integer operations.
// 512 blocks of 16^3 x 16 float32: 14.48 -> 2.10 ms; 64 blocks of 8 x 8 x 32
// float64: 15.04 -> 1.73 ms (before: all of it in FP64, the eigensolve in one warp).
#include "dls_device.cuh"

namespace dls {
namespace {

constexpr int kThreads = 256;
constexpr int kRC = 256;  // rows per staged chunk of the Gram pass

__device__ __forceinline__ double dmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double dadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double dsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double ddiv(double a, double b) { return __ddiv_rn(a, b); }
__device__ __forceinline__ double dfma(double a, double b, double c) { return __fma_rn(a, b, c); }

template <typename T> __device__ __forceinline__ double to_dt(double x);
template <> __device__ __forceinline__ double to_dt<float>(double x) { return (double)__double2float_rn(x); }
template <> __device__ __forceinline__ double to_dt<double>(double x) { return x; }

// Dequantized coefficient in the field dtype: dtype(q) * dtype(delta).
template <typename T> __device__ __forceinline__ T dequant(int32_t q, T delta_t);
template <> __device__ __forceinline__ float dequant<float>(int32_t q, float d) { return __fmul_rn(__int2float_rn(q), d); }
template <> __device__ __forceinline__ double dequant<double>(int32_t q, double d) { return __dmul_rn((double)q, d); }
template <typename T> __device__ __forceinline__ T tfma(T a, T b, T c);
template <> __device__ __forceinline__ float tfma<float>(float a, float b, float c) { return __fmaf_rn(a, b, c); }
template <> __device__ __forceinline__ double tfma<double>(double a, double b, double c) { return __fma_rn(a, b, c); }

// Rotation parameters of one round.
template <int NM>
struct Rot {
  double c[NM / 2], s[NM / 2], t[NM / 2];
  int pq[NM / 2];            // p | q << 8 | active << 16
  int pair_of[NM];
  int any;
};

template <typename T, int NM>
struct Smem {
  static constexpr int LD = NM + 1;      // odd row length: rows and columns of doubles spread over the banks
  double G[2][NM * LD], V[NM * LD];
  // Gram chunk (kRC x n), E(r) residuals of a chunk, or every thread's E(r)
  // estimates (floats, [r][thread])
  double buf[kRC * LD];
  double part[kRC / 32 * NM];
  double colsum[NM];
  alignas(16) T Vt[NM * NM];             // stored modes, Vt[k * NM + j] = Vst[j][k], zeros for j >= n
  Rot<NM> rot[2];
  int64_t coff[NM];                      // field offset of column j
  double tol, Ecur;
  float Eest[NM + 1];
  int ovf, nonfinite, no_est;
  int wq[NM];
  int ncorr, nesc, kmax;
};

// Field offset of the block's spatial point ls (x fastest): extents are small.
__device__ __forceinline__ int64_t spatial_off(const Plan& P, const Geom& g, uint32_t ls) {
  const uint32_t sx = (uint32_t)g.sx, r = ls / sx, x = ls - r * sx;
  const uint32_t z = r / (uint32_t)g.sy, y = r - z * (uint32_t)g.sy;
  return (int64_t)z * (P.dims[0] * P.dims[1]) + (int64_t)y * P.dims[0] + x;
}
// A[l][j] = in[block_base + row_off(l) + coff[j]].
__device__ __forceinline__ int64_t block_base(const Plan& P, const Geom& g) {
  return (int64_t)g.v * P.K + g.t0 * P.P + g.z0 * (P.dims[0] * P.dims[1]) + g.y0 * P.dims[0] + g.x0;
}
__device__ __forceinline__ int64_t row_off(const Plan& P, const Geom& g, int64_t l) {
  return g.side == 0 ? spatial_off(P, g, (uint32_t)l) : l * P.P;
}

// Round-robin pairing (circle method) of m indices, round `round`, pair i.
__device__ __forceinline__ void rr_pair(int round, int i, int m, int& p, int& q) {
  int a, b;
  if (i == 0) { a = m - 1; b = round; }
  else {
    a = round + i;
    a = a >= m - 1 ? a - (m - 1) : a;
    b = round - i;
    b = b < 0 ? b + (m - 1) : b;
  }
  p = a < b ? a : b;
  q = a < b ? b : a;
}

// Rotations of a round from the matrix at its start (warp 0, a lane a pair).
template <int NM>
__device__ void rotations(const double* G, Rot<NM>& R, int round, int n, int m, double tol, int lane) {
  constexpr int LD = NM + 1;
  int act = 0;
  if (lane < m / 2) {
    int p, q;
    rr_pair(round, lane, m, p, q);
    if (q < n) {
      const double apq = G[p * LD + q];
      if (mag_above(apq, tol) && !mag_above(apq, INFINITY)) {
        // tests on the bit patterns; reciprocals round as the quotients 1 / x
        const double theta = ddiv(dsub(G[q * LD + q], G[p * LD + p]), dmul(2.0, apq));
        double t;
        if (mag_above(theta, 1e150)) {
          t = ddiv(0.5, theta);
        } else {
          t = __drcp_rn(dadd(fabs(theta), __dsqrt_rn(dadd(1.0, dmul(theta, theta)))));
          const long long tb = __double_as_longlong(theta);
          if (tb < 0 && (tb << 1) != 0) t = -t;          // theta < 0
        }
        const double c = __drcp_rn(__dsqrt_rn(dadd(1.0, dmul(t, t))));
        R.c[lane] = c;
        R.s[lane] = dmul(t, c);
        R.t[lane] = t;
        act = 1;
      }
      R.pair_of[q] = lane;
    }
    R.pair_of[p] = lane;
    R.pq[lane] = p | q << 8 | act << 16;
  }
  const unsigned any = __ballot_sync(0xffffffffu, act);
  if (lane == 0) R.any = any != 0u;
}

// Jacobi eigensolve of S.G[0] (n x n), all threads; eigenvectors in S.V
// (unsorted), eigenvalues on the diagonal of the returned buffer.  Mirrors the
// definition step by step: rotations of a round are computed from the matrix
// at the start of the round, rows are rotated, then columns, the upper
// triangle is mirrored, and the rotated pairs get their closed-form diagonal
// and a zero off-diagonal.  An upper-triangle entry (a, b) depends on four
// entries of the old matrix (a's pair by b's pair), so a thread forms each
// entry on its own, from one buffer into the other; a rotation with its factor
// signs folded in (x1 u + x2 w, x2 = -s) rounds as the definition's
// difference, and the operands are selected so that every lane runs the same
// nine operations (an FP64 instruction holds its quarter of the SM for 64
// clocks however few lanes take part).  Warp 0 works out the next round's
// rotations while the other warps rotate the columns of V.
// Bound by the FP64 pipe (6 operations an entry of V's active pairs, up to 9
// an entry of G's triangle) and, with one CTA on an SM, by the chain of
// divisions and square roots of a rotation (560 and 600 clocks each).  (One warp with a row a lane took
// 32-way bank conflicts: 15 ms for 64 matrices of order 32.)
template <typename T, int NM>
__device__ int jacobi_block(Smem<T, NM>& S, int n) {
  constexpr int LD = NM + 1;
  constexpr int kSlots = (NM * (NM + 1) / 2 + kThreads - 1) / kThreads;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int m = n + (n & 1), h = m / 2;
  int ea[kSlots], eb[kSlots];              // this thread's upper-triangle entries
#pragma unroll
  for (int s = 0; s < kSlots; ++s) {
    int idx = tid + s * kThreads;
    ea[s] = -1;
    eb[s] = 0;
    if (idx < n * (n + 1) / 2) {
      int i = 0;
      while (idx >= n - i) { idx -= n - i; ++i; }
      ea[s] = i;
      eb[s] = i + idx;
    }
  }
  for (int e = tid; e < n * n; e += kThreads) {
    const int a = e / n, b = e - a * n;
    S.V[a * LD + b] = a == b ? 1.0 : 0.0;
  }
  if (tid == 0) {
    double tr = 0.0;
    for (int i = 0; i < n; ++i) tr = dadd(tr, S.G[0][i * LD + i]);
    S.tol = dmul(1e-15, tr);
  }
  __syncthreads();
  const double tol = S.tol;
  int cur = 0, pb = 0;
  if (n > 1) {
    if (warp == 0) rotations<NM>(S.G[0], S.rot[0], 0, n, m, tol, lane);
    __syncthreads();
  }
  for (int sweep = 0; sweep < 30 && n > 1; ++sweep) {
    int rotated = 0;
    for (int round = 0; round < m - 1; ++round) {
      const Rot<NM>& R = S.rot[pb];
      const int any = R.any;
      if (any) {
        rotated = 1;
        const double* G = S.G[cur];
        double* G2 = S.G[cur ^ 1];
#pragma unroll
        for (int s = 0; s < kSlots; ++s) {
          if (tid - lane + s * kThreads >= n * (n + 1) / 2) break;     // no entry in this warp
          const bool on = ea[s] >= 0;
          const int a = on ? ea[s] : 0, b = on ? eb[s] : 0;
          const int ka = R.pair_of[a], kb = R.pair_of[b];
          const int wa = R.pq[ka], wb = R.pq[kb];
          const bool acta = (wa >> 16) != 0, actb = (wb >> 16) != 0, own = ka == kb && acta;
          const int pa = wa & 255, qa = (wa >> 8) & 255, p = wb & 255, q = (wb >> 8) & 255;
          const bool first = a == pa;
          double v = G[a * LD + b];
          // the rotated pair's own diagonal: 1 G[a][a] -+ t G[p][q], in the same operations
          const double ca = R.c[ka], sa = R.s[ka], ta = R.t[ka];
          const double x1 = own ? 1.0 : (first ? ca : sa), x2 = own ? (first ? -ta : ta) : (first ? -sa : ca);
          // entries (a, cp) and (a, q) of the row rotation: b's pair, or b alone where it rests
          const int cp = actb ? p : b, cq = actb ? q : b, rq = acta ? qa : a, rp = acta ? pa : a;
          double hp = G[a * LD + cp], hq = G[a * LD + cq];
          if (__any_sync(0xffffffffu, acta)) {
            const double up = own ? v : G[rp * LD + cp], wp = own ? G[p * LD + q] : G[rq * LD + cp];
            const double ep = dadd(dmul(x1, up), dmul(x2, wp));
            hp = acta ? ep : hp;
            if (__any_sync(0xffffffffu, acta && actb && !own)) {
              const double eq = dadd(dmul(x1, G[rp * LD + cq]), dmul(x2, G[rq * LD + cq]));
              hq = acta ? eq : hq;
            }
            if (acta && !actb) v = hp;
          }
          if (__any_sync(0xffffffffu, actb && !own)) {
            const double cb = R.c[kb], sb = R.s[kb];
            const double y1 = b == p ? cb : sb, y2 = b == p ? -sb : cb;
            const double rv = dadd(dmul(y1, hp), dmul(y2, hq));
            v = actb && !own ? rv : v;
          }
          if (own) v = a == b ? hp : 0.0;
          if (on) {
            G2[a * LD + b] = v;
            G2[b * LD + a] = v;
          }
        }
        cur ^= 1;
        __syncthreads();
      }
      const int next = round + 1 < m - 1 ? round + 1 : 0;
      if (warp == 0) {
        rotations<NM>(S.G[cur], S.rot[pb ^ 1], next, n, m, tol, lane);
      } else if (any && (warp & 3) != 0) {
        // (warp 4 shares warp 0's FP64 unit: its chain of divisions is the longer side)
        const int vt = (warp - 1 - (warp > 4 ? 1 : 0)) * 32 + lane;
        for (int it = vt; it < n * h; it += 6 * 32) {
          const int a = it / h, i = it - a * h;
          const int w = R.pq[i];
          if (!(w >> 16)) continue;
          const int p = w & 255, q = (w >> 8) & 255;
          const double c = R.c[i], sn = R.s[i];
          const double vp = S.V[a * LD + p], vq = S.V[a * LD + q];
          S.V[a * LD + p] = dsub(dmul(c, vp), dmul(sn, vq));
          S.V[a * LD + q] = dadd(dmul(sn, vp), dmul(c, vq));
        }
      }
      __syncthreads();
      pb ^= 1;
    }
    if (!rotated) break;
  }
  return cur;
}

// Stable descending order of the clamped eigenvalues, sign-normalised
// columns, first rcap columns rounded to the dtype into S.Vt (warp 0).
template <typename T, int NM>
__device__ void sort_and_store(Smem<T, NM>& S, const double* G, int n, int rcap, int lane, double* vst_out) {
  constexpr int LD = NM + 1;
  if (lane < n) {
    const int k = lane;
    double dk = G[k * LD + k];
    dk = dk < 0.0 ? 0.0 : dk;
    int pos = 0;
    for (int j = 0; j < n; ++j) {
      double dj = G[j * LD + j];
      dj = dj < 0.0 ? 0.0 : dj;
      if (dj > dk || (dj == dk && j < k)) ++pos;
    }
    int imax = 0;
    double amax = -1.0;
    for (int a = 0; a < n; ++a) {
      double av = fabs(S.V[a * LD + k]);
      if (av > amax) { amax = av; imax = a; }
    }
    const bool neg = S.V[imax * LD + k] < 0.0;
    if (pos < rcap) {
      for (int a = 0; a < n; ++a) {
        double v = S.V[a * LD + k];
        v = neg ? -v : v;
        const double vs = to_dt<T>(v);
        S.Vt[pos * NM + a] = (T)vs;
        vst_out[a * rcap + pos] = vs;
      }
    }
  }
}

// E(r) = sum (A - D_r)^2 in the fixed order: per column, rows in chunks of 32
// (sequential fma), chunk sums in order, then column sums in order.
// D_r is the decode contract: fma chain over k < r in the field dtype.
// Rows kRC at a time: their residuals (independent) into shared memory, then a
// thread per chunk and column for the ordered sums.
template <typename T, int NM>
__device__ __noinline__ double block_err(Smem<T, NM>& S, const Plan& P, const Geom& g, const T* __restrict__ in,
                                         const int32_t* __restrict__ q, int r, T delta_t) {
  constexpr int LD = NM + 1;
  const int tid = threadIdx.x, n = g.n;
  const int64_t L = g.L, base = block_base(P, g);
  if (tid < n) S.colsum[tid] = 0.0;
  __syncthreads();
  for (int64_t l0 = 0; l0 < L; l0 += kRC) {
    const int rows = (int)((L - l0) < kRC ? (L - l0) : kRC);
    const int ncg = rows >= kThreads ? 1 : (kThreads / rows < n ? kThreads / rows : n);   // column groups
    for (int it = tid; it < rows * ncg; it += kThreads) {
      const int cg = it / rows, lr = it - cg * rows;
      const int64_t l = l0 + lr;
      T ch[NM];
#pragma unroll
      for (int k = 0; k < NM; ++k) ch[k] = (k < r) ? dequant<T>(q[(int64_t)k * L + l], delta_t) : T(0);
      const T* row = in + base + row_off(P, g, l);
      for (int j = cg; j < n; j += ncg) {
        T acc = T(0);
#pragma unroll
        for (int k = 0; k < NM; ++k)
          if (k < r) acc = tfma<T>(ch[k], S.Vt[k * NM + j], acc);
        S.buf[lr * LD + j] = dsub(widen(row[S.coff[j]]), widen_any(acc));   // (an infinite acc makes E infinite)
      }
    }
    __syncthreads();
    const int nch = (rows + 31) / 32;
    for (int it = tid; it < nch * n; it += kThreads) {
      const int c = it / n, j = it - c * n;
      const int e = (c + 1) * 32 < rows ? (c + 1) * 32 : rows;
      double pc = 0.0;
      for (int lr = c * 32; lr < e; ++lr) {
        const double d = S.buf[lr * LD + j];
        pc = dfma(d, d, pc);
      }
      S.part[c * NM + j] = pc;
    }
    __syncthreads();
    if (tid < n) {
      double s = S.colsum[tid];
      for (int c = 0; c < nch; ++c) s = dadd(s, S.part[c * NM + tid]);
      S.colsum[tid] = s;
    }
  }
  __syncthreads();
  if (tid == 0) {
    double E = 0.0;
    for (int j = 0; j < n; ++j) E = dadd(E, S.colsum[j]);
    S.Ecur = E;
  }
  __syncthreads();
  const double E = S.Ecur;
  __syncthreads();
  return E;
}

// One coefficient by the definition: c = fma chain over j, q = rint(c / delta).
template <typename T, int NM>
__device__ __noinline__ int32_t coeff_exact(const Smem<T, NM>& S, const T* row, int n, int k, double delta,
                                            double qlim, int* ovf) {
  double c = 0.0;
  for (int j = 0; j < n; ++j) c = dfma(widen(row[S.coff[j]]), widen(S.Vt[k * NM + j]), c);
  const double y = ddiv(c, delta);
  if (!(fabs(y) < qlim)) { *ovf = 1; return 0; }
  return (int32_t)rint(y);
}

// q = rint(c / delta) of an FP64 coefficient: from c (1 / delta) where that
// product is clear of a half-integer by more than its error (a few units in
// the last place), else from the quotient.
__device__ __noinline__ int32_t quot_exact(double c, double delta, double qlim, int* ovf) {
  const double y = ddiv(c, delta);
  if (!(fabs(y) < qlim)) { *ovf = 1; return 0; }
  return (int32_t)rint(y);
}
__device__ __forceinline__ int32_t quot(double c, double delta, double inv, bool inv_ok, double qlim, int* ovf) {
  constexpr double kMagic = 6755399441055744.0;        // 1.5 x 2^52: y + kMagic rounds y to an integer
  const double y = dmul(c, inv);
  if (inv_ok && mag_below(y, 1.0e9)) {                  // below qlim = 2^30, and |y| 2^-50 < 1e-6
    const double z = dadd(y, kMagic);
    const double f = dsub(y, dsub(z, kMagic));
    if (mag_below(f, 0.499999)) return __double2loint(z);
  }
  return quot_exact(c, delta, qlim, ovf);
}

// The pointwise correction of one value by the definition: k (0 if none) or kEscape.
template <typename T>
__device__ __noinline__ int32_t corr_def(T xv, T xh, double eb, double step, T step_t) {
  const double x = (double)xv;
  const double kk = rint(ddiv(dsub(x, (double)xh), step));
  double xt;
  if (kk == 0.0) xt = (double)xh;
  else if (fabs(kk) > kKmax) return kEscape;
  else xt = (double)tfma<T>((T)kk, step_t, xh);
  if (fabs(dsub(x, xt)) > eb) return kEscape;
  return (int32_t)kk;
}

// The same with the definition left to what needs it.  A residual below the
// bound by more than its rounding needs no correction; on float32 fields one
// whose FP32 quotient is clear of a half-integer (5e-7 relative covers its
// three roundings) and whose corrected value is within the bound by more than
// its rounding is settled too.
struct CorrF {
  double eb, step, eb_lo;
  float step_f, inv_step, eb_lo_f;
  bool ok;                   // the FP32 constants are usable
};
__device__ __forceinline__ int32_t corr_of(float x, float xh, const CorrF& c) {
  if (c.ok) {
    const float R = __fsub_rn(x, xh);
    if (fabsf(R) < c.eb_lo_f) return 0;
    const float y = __fmul_rn(R, c.inv_step), k = rintf(y);
    if (fabsf(__fsub_rn(y, k)) < 0.5f - (__fmul_rn(fabsf(y), 5.0e-7f) + 1.0e-30f) && fabsf(k) <= 1048576.0f &&
        fabsf(__fsub_rn(x, __fmaf_rn(k, c.step_f, xh))) <= c.eb_lo_f)
      return (int32_t)k;
  }
  return corr_def<float>(x, xh, c.eb, c.step, c.step_f);
}
__device__ __forceinline__ int32_t corr_of(double x, double xh, const CorrF& c) {
  if (mag_below(dsub(x, xh), c.eb_lo)) return 0;
  return corr_def<double>(x, xh, c.eb, c.step, c.step);
}

// Projection, quantization and FP32 estimates of every E(r) of a float32
// block, a row a thread: q[k][l] = rint((sum_j A[l][j] Vst[j][k]) / delta).
// The FP32 coefficient is within 18 u |row| of the FP64 chain (16 products; 34
// for 32) and its quotient within 3 u |y| more, so it settles q where it is
// clear of a half-integer by that much.  The decoded row is the decode
// contract's own, so an estimate of E(r) carries the roundings of its sum of
// non-negative terms alone.
template <int NM>
__device__ void project_f32(Smem<float, NM>& S, const Plan& P, const Geom& g, const float* __restrict__ in,
                            int32_t* __restrict__ qb, int rcap, double delta, float delta_t, bool filt, int* ovf) {
  const int tid = threadIdx.x, n = g.n;
  const int64_t L = g.L, base = block_base(P, g);
  float* E = reinterpret_cast<float*>(S.buf);           // [r][thread]
  static_assert(sizeof(S.buf) >= sizeof(float) * (NM + 1) * kThreads, "estimates");
  for (int r = 0; r <= rcap; ++r) E[r * kThreads + tid] = 0.0f;
  const float inv = filt ? __double2float_rn(1.0 / delta) : 0.0f;
  constexpr float kRow = (NM == 16 ? 18.0f : 34.0f) * 1.02f * 5.9604645e-8f;
  bool bad_est = false;
  for (int64_t l = tid; l < L; l += kThreads) {
    const float* row = in + base + row_off(P, g, l);
    float x[NM], acc[NM];
    float n2 = 0.0f;
#pragma unroll
    for (int j = 0; j < NM; ++j) x[j] = j < n ? row[S.coff[j]] : 0.0f;
#pragma unroll
    for (int j = 0; j < NM; ++j) {
      acc[j] = 0.0f;
      n2 = __fmaf_rn(x[j], x[j], n2);
    }
    E[tid] += n2;
    // squares that neither overflow nor lose their bits (an all-zero row is exact)
    float amax = 0.0f;
#pragma unroll
    for (int j = 0; j < NM; ++j) amax = fmaxf(amax, fabsf(x[j]));
    const bool row_ok = filt && n2 < 1.0e36f && (n2 > 1.0e-30f || amax == 0.0f);
    if (!(n2 < 1.0e36f)) bad_est = true;
    const float mrow = __fmul_rn(__fmul_rn(sqrtf(n2), 1.0001f * kRow), inv);
#pragma unroll 1
    for (int k = 0; k < rcap; ++k) {
      const float4* vp = reinterpret_cast<const float4*>(&S.Vt[k * NM]);
      float v[NM];
#pragma unroll
      for (int j4 = 0; j4 < NM / 4; ++j4) {
        const float4 t = vp[j4];
        v[4 * j4 + 0] = t.x; v[4 * j4 + 1] = t.y; v[4 * j4 + 2] = t.z; v[4 * j4 + 3] = t.w;
      }
      float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f, s3 = 0.0f;
#pragma unroll
      for (int j = 0; j < NM; j += 4) {
        s0 = __fmaf_rn(x[j], v[j], s0);
        s1 = __fmaf_rn(x[j + 1], v[j + 1], s1);
        s2 = __fmaf_rn(x[j + 2], v[j + 2], s2);
        s3 = __fmaf_rn(x[j + 3], v[j + 3], s3);
      }
      const float y = __fmul_rn(__fadd_rn(__fadd_rn(s0, s1), __fadd_rn(s2, s3)), inv);
      const float ry = rintf(y);
      const float mar = __fadd_rn(mrow, __fmaf_rn(fabsf(y), 4.0e-7f, 1.0e-30f));
      int32_t qv;
      if (row_ok && fabsf(__fsub_rn(y, ry)) < 0.5f - mar && fabsf(y) < 1.6e7f) qv = (int32_t)ry;
      else qv = coeff_exact<float, NM>(S, row, n, k, delta, kQmaxF32, ovf);
      qb[(int64_t)k * L + l] = qv;
      const float ch = dequant<float>(qv, delta_t);
      float e0 = 0.0f, e1 = 0.0f;
#pragma unroll
      for (int j = 0; j < NM; j += 2) {
        acc[j] = __fmaf_rn(ch, v[j], acc[j]);
        acc[j + 1] = __fmaf_rn(ch, v[j + 1], acc[j + 1]);
        const float d0 = __fsub_rn(x[j], acc[j]), d1 = __fsub_rn(x[j + 1], acc[j + 1]);
        e0 = __fmaf_rn(d0, d0, e0);
        e1 = __fmaf_rn(d1, d1, e1);
      }
      E[(k + 1) * kThreads + tid] += __fadd_rn(e0, e1);
    }
  }
  if (bad_est) S.no_est = 1;
  __syncthreads();
  const int lane = tid & 31, warp = tid >> 5;
  for (int r = warp; r <= rcap; r += kThreads / 32) {
    float s = 0.0f;
    for (int t = lane; t < kThreads; t += 32) s = __fadd_rn(s, E[r * kThreads + t]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s = __fadd_rn(s, __shfl_xor_sync(0xffffffffu, s, o));
    if (lane == 0) S.Eest[r] = s;
  }
}

// Projection and quantization of a float64 block: the FP64 chain of every
// coefficient (a row a thread, or a row and a group of columns where the block
// has fewer rows than the CTA has threads).
template <int NM>
__device__ void project_f64(Smem<double, NM>& S, const Plan& P, const Geom& g, const double* __restrict__ in,
                            int32_t* __restrict__ qb, int rcap, double delta, int* ovf) {
  const int n = g.n;
  const int64_t L = g.L, base = block_base(P, g);
  const int kg = L >= kThreads || rcap == 0 ? 1 : ((int)(kThreads / L) < rcap ? (int)(kThreads / L) : rcap);
  const double inv = ddiv(1.0, delta);
  const bool inv_ok = inv < 1e300 && inv > 1e-300;
  for (int64_t it = threadIdx.x; it < L * kg; it += kThreads) {
    const int k0 = (int)(it / L);
    const int64_t l = it - k0 * L;
    const double* row = in + base + row_off(P, g, l);
    double a[NM];
#pragma unroll
    for (int j = 0; j < NM; ++j) a[j] = j < n ? row[S.coff[j]] : 0.0;
    for (int k = k0; k < rcap; k += kg) {
      double c = 0.0;
#pragma unroll
      for (int j = 0; j < NM; ++j)
        if (j < n) c = dfma(a[j], S.Vt[k * NM + j], c);
      qb[(int64_t)k * L + l] = quot(c, delta, inv, inv_ok, kQmaxF64, ovf);
    }
  }
}

template <typename T, int NM>
__global__ void __launch_bounds__(kThreads, 2) k_plain(Plan P, const T* __restrict__ in, Work W) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem<T, NM>& S = *reinterpret_cast<Smem<T, NM>*>(smem_raw);
  constexpr int LD = NM + 1;
  const int64_t bi = blockIdx.x;
  const Geom g = block_geom(P, P.b0 + bi);
  const VarInfo vi = W.vars[g.v];
  const int n = g.n;
  const int64_t L = g.L, N = g.N, base = block_base(P, g);
  const int rcap = P.rank_cap < n ? P.rank_cap : n;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const T delta_t = (T)to_dt<T>(vi.delta);

  if (tid == 0) { S.ovf = 0; S.nonfinite = 0; S.no_est = 0; S.ncorr = 0; S.nesc = 0; S.kmax = 0; }
  if (tid < NM) {
    S.wq[tid] = 0;
    S.coff[tid] = tid < n ? (g.side == 0 ? tid * P.P : spatial_off(P, g, tid)) : 0;
  }
  for (int e = tid; e < NM * NM; e += kThreads) S.Vt[e] = T(0);
  __syncthreads();

  // ---- 1. Gram: G[i][j] = sum_l A[l][i] A[l][j], sequential fma over l
  const int npairs = n * (n + 1) / 2;
  constexpr int kPairsPerThread = (NM * (NM + 1) / 2 + kThreads - 1) / kThreads;
  double acc[kPairsPerThread];
  int pi[kPairsPerThread], pj[kPairsPerThread];
#pragma unroll
  for (int s = 0; s < kPairsPerThread; ++s) {
    acc[s] = 0.0;
    int idx = tid + s * kThreads;
    pi[s] = -1; pj[s] = -1;
    if (idx < npairs) {
      int i = 0;
      while (idx >= n - i) { idx -= n - i; ++i; }
      pi[s] = i; pj[s] = i + idx;
    }
  }
  int nonfinite = 0;
  for (int64_t l0 = 0; l0 < L; l0 += kRC) {
    const int rows = (int)((L - l0) < kRC ? (L - l0) : kRC);
    const int ncg = rows >= kThreads ? 1 : (kThreads / rows < n ? kThreads / rows : n);   // column groups
    for (int it = tid; it < rows * ncg; it += kThreads) {
      const int cg = it / rows, lr = it - cg * rows;
      const T* row = in + base + row_off(P, g, l0 + lr);
#pragma unroll 4
      for (int j = cg; j < n; j += ncg) {
        const T x = row[S.coff[j]];
        if (not_finite(x)) nonfinite = 1;
        S.buf[lr * LD + j] = widen(x);
      }
    }
    __syncthreads();
#pragma unroll
    for (int s = 0; s < kPairsPerThread; ++s) {
      if (pi[s] >= 0) {
        const double* bi_ = S.buf + pi[s];
        const double* bj_ = S.buf + pj[s];
        double a = acc[s];
#pragma unroll 8
        for (int lr = 0; lr < rows; ++lr) a = dfma(bi_[lr * LD], bj_[lr * LD], a);
        acc[s] = a;
      }
    }
    __syncthreads();
  }
  if (nonfinite) S.nonfinite = 1;
#pragma unroll
  for (int s = 0; s < kPairsPerThread; ++s)
    if (pi[s] >= 0) { S.G[0][pi[s] * LD + pj[s]] = acc[s]; S.G[0][pj[s] * LD + pi[s]] = acc[s]; }
  __syncthreads();
  if (S.nonfinite) {
    if (tid == 0) atomicOr(&W.status->nonfinite, 1u);
    return;
  }

  // ---- 2. eigensolve and stored basis; with a fixed basis of this Gram order
  // (Sec. 4), its first rcap modes in the given order instead
  double* vst_out = W.vst + bi * (int64_t)P.nmax * P.nmax;
  if (W.basis && n == P.basis_n) {
    for (int e = tid; e < n * rcap; e += kThreads) {
      const int a = e / rcap, k = e - a * rcap;
      const double vs = to_dt<T>(W.basis[a * n + k]);
      S.Vt[k * NM + a] = (T)vs;
      vst_out[a * rcap + k] = vs;
    }
  } else {
    const int cur = jacobi_block<T, NM>(S, n);
    if (warp == 0) sort_and_store<T, NM>(S, S.G[cur], n, rcap, lane, vst_out);
  }
  __syncthreads();

  // ---- 3. projection and quantization
  int32_t* qb = W.q + (g.pt_off - P.pt_base);
  const double el2 = (P.eb_type == DLS_EB_NRMSE)
                         ? dmul(dmul(vi.eb, vi.eb), ddiv((double)N, P.kbound))
                         : dmul(dmul(vi.eb, vi.eb), (double)N);
  int ovf = 0;
  const bool filt = vi.delta > 1e-30 && vi.delta < 1e30;
  if constexpr (sizeof(T) == 4) project_f32<NM>(S, P, g, in, qb, rcap, vi.delta, delta_t, filt, &ovf);
  else project_f64<NM>(S, P, g, in, qb, rcap, vi.delta, &ovf);
  if (ovf) S.ovf = 1;
  __syncthreads();
  const bool overflow = S.ovf != 0;

  // ---- 4. rank: bisection on pass(r) <=> E(r) <= eps_l^2.  On float32 blocks
  // the FP32 estimate decides where it is clear of eps_l^2 by more than the
  // roundings of its sum (rows a thread x n terms, then the threads').
  const double bnd = (double)(cdiv(L, kThreads) * NM + 80) * 6.6e-8;
  const bool est = sizeof(T) == 4 && !S.no_est && el2 > 1e-30 && bnd < 0.05;
  auto pass = [&](int r) -> bool {
    if (est) {
      const double E = (double)S.Eest[r];
      if (E < 1e37) {
        if (E * (1.0 + 1.1 * bnd) + 1e-36 < el2 * (1.0 - 1e-9)) return true;
        if (E * (1.0 - 1.1 * bnd) - 1e-36 > el2 * (1.0 + 1e-9)) return false;
      }
    }
    return block_err<T, NM>(S, P, g, in, qb, r, delta_t) <= el2;
  };
  int r = 0, nprobes = 0;
  bool raw = overflow;
  if (!raw) {
    int lo = 0, hi = rcap;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      ++nprobes;
      if (pass(mid)) hi = mid; else lo = mid + 1;
    }
    r = lo;
    if (P.eb_type == DLS_EB_NRMSE && !pass(r)) raw = true;
  }

  // ---- 5. pointwise correction at r, and per-block widths
  int32_t* kb = W.kc + (g.pt_off - P.pt_base);
  uint32_t qmx[NM];
#pragma unroll
  for (int k = 0; k < NM; ++k) qmx[k] = 0;
  if (!raw && P.eb_type != DLS_EB_NRMSE) {
    CorrF cf;
    cf.eb = vi.eb;
    cf.step = vi.step;
    cf.eb_lo = vi.eb * (1.0 - 1e-12);
    cf.step_f = __double2float_rn(vi.step);
    cf.ok = vi.eb > 1e-30 && vi.eb < 1e30;
    cf.inv_step = cf.ok ? __double2float_rn(1.0 / vi.step) : 0.0f;
    cf.eb_lo_f = cf.ok ? __double2float_rd(vi.eb * (1.0 - 1e-6)) : 0.0f;
    int nc = 0, ne = 0;
    uint32_t kmx = 0;
    const int64_t es_l = g.side == 0 ? 1 : g.M, es_j = g.side == 0 ? g.M : 1;
    const int ncg = L >= kThreads ? 1 : ((int)(kThreads / L) < n ? (int)(kThreads / L) : n);   // column groups
    for (int64_t it = tid; it < L * ncg; it += kThreads) {
      const int cg = (int)(it / L);
      const int64_t l = it - cg * L;
      T ch[NM];
#pragma unroll
      for (int k = 0; k < NM; ++k) {
        const int32_t qv = (k < r) ? qb[(int64_t)k * L + l] : 0;
        const uint32_t z = zigzag(qv);
        qmx[k] = z > qmx[k] ? z : qmx[k];
        ch[k] = (k < r) ? dequant<T>(qv, delta_t) : T(0);
      }
      const T* row = in + base + row_off(P, g, l);
      int32_t* kr = kb + l * es_l;
#pragma unroll 2
      for (int j = cg; j < n; j += ncg) {
        T xh = T(0);
#pragma unroll
        for (int k = 0; k < NM; ++k)
          if (k < r) xh = tfma<T>(ch[k], S.Vt[k * NM + j], xh);
        const int32_t kv = corr_of(row[S.coff[j]], xh, cf);
        if (kv == kEscape) {
          ++ne;
        } else if (kv != 0) {
          ++nc;
          const uint32_t z = zigzag(kv);
          kmx = z > kmx ? z : kmx;
        }
        kr[j * es_j] = kv;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      nc += __shfl_xor_sync(0xffffffffu, nc, o);
      ne += __shfl_xor_sync(0xffffffffu, ne, o);
      kmx = max(kmx, __shfl_xor_sync(0xffffffffu, kmx, o));
    }
    if (lane == 0) {
      atomicAdd(&S.ncorr, nc);
      atomicAdd(&S.nesc, ne);
      atomicMax(&S.kmax, (int)kmx);
    }
  } else if (!raw) {
    // NRMSE mode: no corrections, widths only
    for (int64_t l = tid; l < L; l += kThreads) {
#pragma unroll
      for (int k = 0; k < NM; ++k)
        if (k < r) { uint32_t z = zigzag(qb[(int64_t)k * L + l]); qmx[k] = z > qmx[k] ? z : qmx[k]; }
    }
    for (int64_t e = tid; e < N; e += kThreads) kb[e] = 0;
  }
  if (!raw) {
#pragma unroll
    for (int k = 0; k < NM; ++k) {
      if (k < r) {
        const uint32_t v = __reduce_max_sync(0xffffffffu, qmx[k]);
        if (lane == 0) atomicMax(&S.wq[k], bit_width(v));
      }
    }
  }
  __syncthreads();

  // ---- 6. record size (raw when the encoded record is not smaller)
  if (tid == 0) {
    BlockMeta m;
    const int es = (int)sizeof(T);
    const int64_t rawsz = raw_record_bytes(N, es);
    m.rcap = rcap;
    m.nprobes = nprobes;
    m.r = 0; m.wk = 0; m.ib = 0; m.ncorr = 0; m.nesc = 0;
    m.flags = g.side ? (int)kFlagSpatial : 0;
    for (int k = 0; k < kMaxN; ++k) m.wq[k] = 0;
    if (!raw) {
      for (int k = 0; k < r; ++k) m.wq[k] = (uint8_t)S.wq[k];
      const int wk = bit_width((uint32_t)S.kmax);
      const int ib = bit_width((uint32_t)(N - 1));
      const RecLayout lay = rec_layout(r, n, L, N, es, m.wq, wk, ib, S.ncorr, S.nesc);
      if (lay.size >= rawsz) {
        raw = true;
      } else {
        m.r = r; m.wk = wk; m.ib = ib; m.ncorr = S.ncorr; m.nesc = S.nesc;
        m.flags |= lay.dense ? (int)kFlagDense : 0;
        m.nbytes = lay.size;
      }
    }
    if (raw) {
      m.r = 0; m.wk = 0; m.ib = 0; m.ncorr = 0; m.nesc = 0;
      for (int k = 0; k < kMaxN; ++k) m.wq[k] = 0;
      m.flags = (int)kFlagRaw | (g.side ? (int)kFlagSpatial : 0);
      m.nbytes = rawsz;
    }
    W.meta[bi] = m;
  }
}

template <typename T, int NM>
int launch_t(const Plan& p, const void* d_in, const Work& w, cudaStream_t s) {
  const size_t smem = sizeof(Smem<T, NM>);
  cudaError_t e = cudaFuncSetAttribute(k_plain<T, NM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return DLS_ERR_CUDA;
  if (p.nb == 0) return DLS_OK;
  k_plain<T, NM><<<(unsigned)p.nb, kThreads, smem, s>>>(p, (const T*)d_in, w);
  return cudaGetLastError() == cudaSuccess ? DLS_OK : DLS_ERR_CUDA;
}

}  // namespace

int launch_plain_compress(const Plan& p, const void* d_in, const Work& w, cudaStream_t s) {
  if (p.dtype == DLS_F32) {
    if (p.nmax <= 16) return launch_t<float, 16>(p, d_in, w, s);
    return launch_t<float, 32>(p, d_in, w, s);
  }
  if (p.nmax <= 16) return launch_t<double, 16>(p, d_in, w, s);
  return launch_t<double, 32>(p, d_in, w, s);
}

}  // namespace dls
