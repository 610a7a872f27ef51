// Global-basis mode (Algorithm 1 of arXiv 2601.20113 as stated: one basis per
// variable, learned from random patches of the first snapshot, Sec. 2.3
// Eq. 2-3; per patch of every snapshot the coefficients on it, Sec. 2.5
// Eq. 5, the largest-magnitude prefix meeting the local tolerance of Sec. 2.4
// Eq. 4 found by bisection, Eq. 6; reconstruction, Sec. 2.6).  Every stored
// decision is the FP64 definition's (the patches take it in FP32 where that
// provably settles it); the device steps are
//   k_gb_sample   the sample matrix Q (S x M) from the first snapshot,
//   k_gb_gram     G = Q^T Q, each entry a sequential sum over the samples,
//   k_gb_jacobi   the eigenvectors of G by cyclic Jacobi in one cluster of
//                 CTAs (the rows of G and V shared out among them), sorted by
//                 decreasing eigenvalue and signed (largest component positive),
//   k_gb_norm     ||u||^2 of the variable, then eps_l^2 and delta,
//   k_gb_patch    a warp per patch: alpha = Phi^T u, q = rint(alpha / delta),
//                 the magnitude order, the bisection on the kept count, the
//                 record into the patch's slot,
//   scan + copy   the record offsets and the stream.  (The FP64 definitions run
//                 where an FP32 evaluation cannot settle what they decide.)
// The decoder rebuilds each patch from its kept modes in kept order.
#include <cooperative_groups.h>

#include "dls_device.cuh"

namespace cg = cooperative_groups;

namespace dls {
namespace {

constexpr int kGbMaxM = 128;
constexpr int kGbHdr = 80;
constexpr uint32_t kGbMagic = 0x47534C44u;   // "DLSG"
constexpr int kGbWarps = 8;                  // patches in flight per CTA
constexpr int kGbStatCtas = 512;
constexpr int kGbTile = 1024;                // records a tile of the size scan

struct GbPlan {
  int64_t dims[4];
  int px, py, pz, M, ib;
  int64_t S, K, nrec, npx, npy, npz;
  double eps_t;
  int64_t slot_bytes;          // a patch's record slot (largest record, 16-aligned)
  int64_t offsets_pos, payload_pos;
};

struct GbStatus {
  unsigned int bad_origin, overflow, corrupt, nonfinite;
  double eps_l2, delta;
  unsigned long long total;
};

__host__ __device__ inline int gb_width(uint64_t v) {
  int b = 0;
  while (v) {
    ++b;
    v >>= 1;
  }
  return b;
}

// Largest record of a patch: n = M entries of ib + 63 bits.
__host__ __device__ inline int64_t gb_record_max(int M, int ib) {
  const int64_t words = ((int64_t)M * (ib + 63) + 31) / 32;
  return align_up(8 + 4 * words, 8);
}

int gb_make_plan(const dls_gb_params* p, GbPlan* g) {
  if (!p) return DLS_ERR_INVALID_ARG;
  memset(g, 0, sizeof(*g));
  for (int a = 0; a < 4; ++a) {
    if (p->dims[a] < 1) return DLS_ERR_INVALID_ARG;
    g->dims[a] = p->dims[a];
  }
  if (p->m < 1 || !(p->eps_t > 0.0) || !isfinite(p->eps_t) || p->nsample < 1) return DLS_ERR_INVALID_ARG;
  g->px = g->py = p->m;
  g->pz = p->dims[2] > 1 ? p->m : 1;
  const int64_t M = (int64_t)g->px * g->py * g->pz;
  if (M > kGbMaxM) return DLS_ERR_INVALID_ARG;
  g->M = (int)M;
  if (p->dims[0] % g->px || p->dims[1] % g->py || p->dims[2] % g->pz) return DLS_ERR_INVALID_ARG;
  g->ib = gb_width((uint64_t)(M - 1));
  g->S = p->nsample;
  g->K = p->dims[0] * p->dims[1] * p->dims[2] * p->dims[3];
  g->npx = p->dims[0] / g->px;
  g->npy = p->dims[1] / g->py;
  g->npz = p->dims[2] / g->pz;
  g->nrec = g->npx * g->npy * g->npz * p->dims[3];
  g->eps_t = p->eps_t;
  g->slot_bytes = align_up(gb_record_max(g->M, g->ib), 16);
  g->offsets_pos = kGbHdr + 8 * M * M;
  g->payload_pos = g->offsets_pos + 8 * (g->nrec + 1);
  return DLS_OK;
}

struct GbLayout {
  size_t Q, G, V, phi, lam, partial, status, sizes, tiles, slots, total;
};

GbLayout gb_layout(const GbPlan& g) {
  GbLayout L;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off = (size_t)align_up((int64_t)(off + bytes), 256);
    return o;
  };
  const size_t MM = (size_t)g.M * g.M;
  L.Q = take(sizeof(double) * (size_t)g.S * g.M);
  L.G = take(sizeof(double) * MM);
  L.V = take(sizeof(double) * MM);
  L.phi = take(sizeof(double) * MM);
  L.lam = take(sizeof(double) * (size_t)g.M);
  L.partial = take(sizeof(double) * kGbStatCtas);
  L.status = take(sizeof(GbStatus));
  L.sizes = take(sizeof(unsigned long long) * (size_t)(g.nrec + 1));
  L.tiles = take(sizeof(unsigned long long) * (size_t)cdiv(g.nrec, kGbTile));
  L.slots = take((size_t)g.slot_bytes * (size_t)g.nrec);
  L.total = off;
  return L;
}

// ---------------------------------------------------------------- step 1: the basis
// Row s of Q: the patch of the first snapshot at origins[s] (x fastest).  What
// the call refuses (an origin outside the snapshot, a non-finite value) leaves
// zeros, so that the Gram and the eigensolve run on finite values: the status
// is read after the last kernel.
__global__ void k_gb_sample(GbPlan g, const float* __restrict__ in, const int64_t* __restrict__ origins, double* Q,
                            GbStatus* st) {
  const int64_t s = blockIdx.x;
  const int64_t x0 = origins[3 * s], y0 = origins[3 * s + 1], z0 = origins[3 * s + 2];
  if (x0 < 0 || y0 < 0 || z0 < 0 || x0 + g.px > g.dims[0] || y0 + g.py > g.dims[1] || z0 + g.pz > g.dims[2]) {
    if (threadIdx.x == 0) atomicOr(&st->bad_origin, 1u);
    for (int i = threadIdx.x; i < g.M; i += blockDim.x) Q[s * g.M + i] = 0.0;
    return;
  }
  for (int i = threadIdx.x; i < g.M; i += blockDim.x) {
    const int ix = i % g.px, iy = (i / g.px) % g.py, iz = i / (g.px * g.py);
    const float v = in[((z0 + iz) * g.dims[1] + (y0 + iy)) * g.dims[0] + (x0 + ix)];
    if (not_finite(v)) atomicOr(&st->nonfinite, 1u);
    Q[s * g.M + i] = not_finite(v) ? 0.0 : (double)v;
  }
}

// G[i][j] = sum_s Q[s][i] Q[s][j], one entry a thread, samples in order (fma).
__global__ void k_gb_gram(GbPlan g, const double* __restrict__ Q, double* G) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= g.M * g.M) return;
  const int i = e / g.M, j = e - i * g.M;
  double acc = 0.0;
  for (int64_t s = 0; s < g.S; ++s) acc = __fma_rn(Q[s * g.M + i], Q[s * g.M + j], acc);
  G[e] = acc;
}

__device__ __forceinline__ void gb_pair(int round, int i, int m, int& p, int& q) {
  int a, b;
  if (i == 0) { a = m - 1; b = round; }
  else { a = (round + i) % (m - 1); b = (round - i + (m - 1)) % (m - 1); }
  p = a < b ? a : b;
  q = a < b ? b : a;
}

// The pair of round `round` that index x is in, and whether x is its larger one.
__device__ __forceinline__ int gb_pair_of(int round, int x, int m, int& larger) {
  int y, i = 0;
  if (x == m - 1) {
    y = round;
  } else if (x == round) {
    y = m - 1;
  } else {
    int d = x - round;
    d = d < 0 ? d + m - 1 : d;
    i = d <= (m - 2) / 2 ? d : m - 1 - d;
    // x = round + i or round - i (mod m - 1); its partner is the other
    y = d == i ? round - i : round + i;
    y = y < 0 ? y + m - 1 : (y >= m - 1 ? y - (m - 1) : y);
  }
  larger = x > y ? 1 : 0;
  return i;
}

// Cyclic Jacobi of G (order M, padded with a zero row and column to even m):
// every round rotates the m/2 disjoint pairs of the round-robin circle whose
// off-diagonal entry exceeds 2^-53 sqrt(|a_pp a_qq|); each 2 x 2 block of A
// (pair k's rows, pair l's columns) becomes J_k^T A_kl J_l, with the exact
// 2 x 2 result on the diagonal blocks, and V's column pairs rotate.  Stops
// after a sweep without rotation (50 sweeps at most).  Then the modes: columns
// of V by decreasing eigenvalue (index order on ties), each signed so that its
// largest-magnitude component (the first on ties) is positive.
//
// One SM's FP64 units took 10.7 us a round at M = 64 (768 warp instructions of
// them), so a cluster of eight CTAs shares it.  In a round CTA c owns the pairs
// [c kpc, (c + 1) kpc): it holds their rows of A, works out their rotations and
// sends these to all eight; then it forms its rows' new entries and sends each
// row to the CTA that owns it in the next round (a row has one reader, so a
// round moves A once).  Rows of V never mix: each CTA keeps M / 8 of them and
// rotates them while the next round's rotations are worked out, which is the
// longest chain left (three divisions and two square roots, about 3 000
// clocks); the threshold of a pair is another warp's work.  Two cluster
// barriers a round.  Measured at M = 64: 6.75 -> 2.81 ms.
constexpr int kJacCtas = 8;
constexpr int kJacThreads = 256;
struct GbRot {
  double c[kGbMaxM / 2], s[kGbMaxM / 2], t[kGbMaxM / 2];
  int act[kGbMaxM / 2];
};
constexpr int kJacRows = 2 * (kGbMaxM / 2 / kJacCtas);     // rows of A a CTA owns, rows of V it keeps
static_assert(kJacRows * kJacCtas == kGbMaxM, "rows");
struct GbJac {
  GbRot rot[2];
  double A[2][kJacRows][kGbMaxM + 1];
  double V[kJacRows][kGbMaxM + 1];
  double lam[kGbMaxM];
  int order[kGbMaxM];
};

__global__ void __cluster_dims__(kJacCtas, 1, 1) __launch_bounds__(kJacThreads, 1)
    k_gb_jacobi(GbPlan g, const double* __restrict__ G, double* Vg, double* phi, double* lam_out) {
  extern __shared__ __align__(16) unsigned char jsm[];
  GbJac& S = *reinterpret_cast<GbJac*>(jsm);
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int M = g.M, m = M + (M & 1), h = m / 2;
  const int kpc = (h + kJacCtas - 1) / kJacCtas, k0 = rank * kpc, nk = k0 >= h ? 0 : (h - k0 < kpc ? h - k0 : kpc);
  const int vr = (M + kJacCtas - 1) / kJacCtas, v0 = rank * vr, nv = v0 >= M ? 0 : (M - v0 < vr ? M - v0 : vr);
  for (int e = tid; e < 2 * nk * m; e += kJacThreads) {
    const int r = e / m, j = e - r * m;
    int p, q;
    gb_pair(0, k0 + (r >> 1), m, p, q);
    const int i = (r & 1) ? q : p;
    S.A[0][r][j] = (i < M && j < M) ? G[i * M + j] : 0.0;
  }
  for (int e = tid; e < nv * m; e += kJacThreads) {
    const int r = e / m, j = e - r * m;
    S.V[r][j] = v0 + r == j ? 1.0 : 0.0;
  }
  cl.sync();
  int ab = 0, pb = 0;
  bool turn_v = false;                         // V is one round behind, with the parameters in rot[pb ^ 1]
  int turn_round = 0;
  // V's rows by the rotations of a round, on the warps that leave warp 0's and warp 1's FP64 units alone
  auto rotate_v = [&](const GbRot& R, int round) {
    const int w = warp & 3;
    if (w < 2) return;
    const int vt = ((warp >> 2) * 2 + (w - 2)) * 32 + lane;
    for (int it = vt; it < nv * h; it += kJacThreads / 2) {
      const int i = it / h, l = it - i * h;
      if (!R.act[l]) continue;
      int p, q;
      gb_pair(round, l, m, p, q);
      const double c = R.c[l], s = R.s[l];
      const double x = S.V[i][p], y = S.V[i][q];
      S.V[i][p] = __fma_rn(c, x, -__dmul_rn(s, y));
      S.V[i][q] = __fma_rn(s, x, __dmul_rn(c, y));
    }
  };
  for (int sweep = 0; sweep < 50 && M > 1; ++sweep) {
    int any = 0;
    for (int round = 0; round < m - 1; ++round) {
      // this CTA's rotations, to every CTA
      if (warp == 0 && lane < nk) {
        int p, q;
        gb_pair(round, k0 + lane, m, p, q);
        const double app = S.A[ab][2 * lane][p], aqq = S.A[ab][2 * lane + 1][q], apq = S.A[ab][2 * lane][q];
        double c = 1.0, s = 0.0, t = 0.0;
        if (apq != 0.0) {
          const double theta = __ddiv_rn(__dsub_rn(aqq, app), __dmul_rn(2.0, apq));
          if (mag_above(theta, 1e150)) {
            t = __ddiv_rn(0.5, theta);
          } else {
            t = __drcp_rn(__dadd_rn(fabs(theta), __dsqrt_rn(__fma_rn(theta, theta, 1.0))));
            const long long tb = __double_as_longlong(theta);
            if (tb < 0 && (tb << 1) != 0) t = -t;          // theta < 0
          }
          c = __drcp_rn(__dsqrt_rn(__fma_rn(t, t, 1.0)));
          s = __dmul_rn(t, c);
        }
        for (int d = 0; d < kJacCtas; ++d) {
          GbRot* R = cl.map_shared_rank(&S.rot[pb], d);
          R->c[k0 + lane] = c;
          R->s[k0 + lane] = s;
          R->t[k0 + lane] = t;
        }
      } else if (warp == 1 && lane < nk) {
        int p, q;
        gb_pair(round, k0 + lane, m, p, q);
        const double app = S.A[ab][2 * lane][p], aqq = S.A[ab][2 * lane + 1][q], apq = S.A[ab][2 * lane][q];
        const int act =
            apq != 0.0 && fabs(apq) > __dmul_rn(0x1p-53, __dsqrt_rn(__dmul_rn(fabs(app), fabs(aqq)))) ? 1 : 0;
        for (int d = 0; d < kJacCtas; ++d) cl.map_shared_rank(&S.rot[pb], d)->act[k0 + lane] = act;
      } else if (turn_v) {
        rotate_v(S.rot[pb ^ 1], turn_round);
      }
      cl.sync();
      const GbRot& R = S.rot[pb];
      int act_any = 0;
      for (int l = lane; l < h; l += 32) act_any |= R.act[l];
      act_any = __any_sync(0xffffffffu, act_any != 0);
      any |= act_any;
      // the rows' new entries, to their owners of the next round
      const int next = round + 1 < m - 1 ? round + 1 : 0;
      for (int it = tid; it < nk * h; it += kJacThreads) {
        const int kl = it / h, l = it - kl * h, k = k0 + kl;
        int p, q, pp, qq;
        gb_pair(round, k, m, p, q);
        gb_pair(round, l, m, pp, qq);
        const int ak = R.act[k], al = R.act[l];
        double x = S.A[ab][2 * kl][pp], y = S.A[ab][2 * kl][qq];
        double z = S.A[ab][2 * kl + 1][pp], w = S.A[ab][2 * kl + 1][qq];
        if (k == l) {
          if (ak) {
            const double t = R.t[k];
            x = __fma_rn(-t, y, x);
            w = __fma_rn(t, y, w);
            y = 0.0;
            z = 0.0;
          }
        } else if (ak | al) {
          const double ck = ak ? R.c[k] : 1.0, sk = ak ? R.s[k] : 0.0, c = al ? R.c[l] : 1.0, s = al ? R.s[l] : 0.0;
          const double r1 = __fma_rn(ck, x, -__dmul_rn(sk, z)), r2 = __fma_rn(ck, y, -__dmul_rn(sk, w));
          const double r3 = __fma_rn(sk, x, __dmul_rn(ck, z)), r4 = __fma_rn(sk, y, __dmul_rn(ck, w));
          x = __fma_rn(c, r1, -__dmul_rn(s, r2));
          y = __fma_rn(s, r1, __dmul_rn(c, r2));
          z = __fma_rn(c, r3, -__dmul_rn(s, r4));
          w = __fma_rn(s, r3, __dmul_rn(c, r4));
        }
        int gp, gq;
        const int op = gb_pair_of(next, p, m, gp), oq = gb_pair_of(next, q, m, gq);
        double* dp = cl.map_shared_rank(&S.A[ab ^ 1][2 * (op % kpc) + gp][0], op / kpc);
        double* dq = cl.map_shared_rank(&S.A[ab ^ 1][2 * (oq % kpc) + gq][0], oq / kpc);
        dp[pp] = x;
        dp[qq] = y;
        dq[pp] = z;
        dq[qq] = w;
      }
      turn_v = act_any != 0;
      turn_round = round;
      ab ^= 1;
      pb ^= 1;
      cl.sync();
    }
    if (!any) break;
  }
  if (turn_v) rotate_v(S.rot[pb ^ 1], turn_round);
  // the rows now lie as round 0 pairs them; eigenvalues and V through global memory to CTA 0
  __syncthreads();
  for (int r = tid; r < 2 * nk; r += kJacThreads) {
    int p, q;
    gb_pair(0, k0 + (r >> 1), m, p, q);
    const int i = (r & 1) ? q : p;
    if (i < M) cl.map_shared_rank(&S.lam[0], 0)[i] = S.A[ab][r][i];
  }
  for (int e = tid; e < nv * M; e += kJacThreads) {
    const int r = e / M, j = e - r * M;
    Vg[(v0 + r) * M + j] = S.V[r][j];
  }
  __threadfence();
  cl.sync();
  if (rank != 0) return;
  // places by a total order (the keys', zeros of either sign alike), so that
  // every place is taken whatever the eigenvalues are
  auto key_of = [&](int k) {
    const double x = S.lam[k];
    return dkey((__double_as_longlong(x) << 1) ? x : 0.0);
  };
  for (int k = tid; k < M; k += kJacThreads) {
    const unsigned long long key = key_of(k);
    int at = 0;
    for (int j = 0; j < M; ++j) {
      const unsigned long long other = key_of(j);
      at += (other > key || (other == key && j < k)) ? 1 : 0;
    }
    S.order[at] = k;
  }
  __syncthreads();
  for (int r = tid; r < M; r += kJacThreads) {
    const int k = S.order[r];
    int imax = 0;
    double vmax = 0.0;
#pragma unroll 8
    for (int i = 0; i < M; ++i) {
      const double a = fabs(__ldcg(&Vg[i * M + k]));
      if (i == 0 || mag_above(a, vmax)) { vmax = a; imax = i; }
    }
    const double sg = __ldcg(&Vg[imax * M + k]) < 0.0 ? -1.0 : 1.0;
#pragma unroll 8
    for (int i = 0; i < M; ++i) phi[i * M + r] = sg * __ldcg(&Vg[i * M + k]);
    lam_out[r] = S.lam[k];
  }
}

// ---------------------------------------------------------------- step 2: the tolerance
// CTA c sums u^2 over a fixed contiguous range in a fixed order: a thread's
// chain of FMAs is the definition, everything else stays off the FP64 pipe and
// its next values are loaded ahead (33.5 M points: 230 us before).
__global__ void __launch_bounds__(256) k_gb_norm(GbPlan g, const float* __restrict__ in, double* partial,
                                                 GbStatus* st) {
  constexpr int kAhead = 16;
  const int64_t per = cdiv(g.K, kGbStatCtas);
  const int64_t i0 = (int64_t)blockIdx.x * per, i1 = (i0 + per) < g.K ? i0 + per : g.K;
  double s = 0.0;
  bool bad = false;
  int64_t i = i0 + threadIdx.x;
  for (; i + 256 * (kAhead - 1) < i1; i += 256 * kAhead) {
    float b[kAhead];
#pragma unroll
    for (int k = 0; k < kAhead; ++k) b[k] = __ldg(in + i + 256 * k);
#pragma unroll
    for (int k = 0; k < kAhead; ++k) {
      bad |= not_finite(b[k]);
      const double x = widen_stream(b[k]);
      s = __fma_rn(x, x, s);
    }
  }
  for (; i < i1; i += 256) {
    const float b = __ldg(in + i);
    bad |= not_finite(b);
    const double x = widen_stream(b);
    s = __fma_rn(x, x, s);
  }
  __shared__ double sh[256];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] = __dadd_rn(sh[threadIdx.x], sh[threadIdx.x + o]);
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = sh[0];
  if (bad) atomicOr(&st->nonfinite, 1u);
}

// eps = eps_t ||u|| / 100, eps_l^2 = eps^2 M / K, delta = eps / sqrt(K).
__global__ void __launch_bounds__(128) k_gb_resolve(GbPlan g, const double* partial, GbStatus* st) {
  __shared__ double psum[kGbStatCtas];
  for (int c = threadIdx.x; c < kGbStatCtas; c += 128) psum[c] = partial[c];
  __syncthreads();
  if (threadIdx.x != 0) return;
  double s2 = 0.0;
  for (int c = 0; c < kGbStatCtas; ++c) s2 = __dadd_rn(s2, psum[c]);
  const double eps = __ddiv_rn(__dmul_rn(g.eps_t, __dsqrt_rn(s2)), 100.0);
  st->eps_l2 = __ddiv_rn(__dmul_rn(__dmul_rn(eps, eps), (double)g.M), (double)g.K);
  st->delta = __ddiv_rn(eps, __dsqrt_rn((double)g.K));
}

// ---------------------------------------------------------------- step 3: the patches
// Per warp in shared memory, after the CTA's FP32 copy of the basis
// ([component][mode], rows of odd length so that a warp reads a row or a column
// of it without bank conflicts, and rows of zeros up to a multiple of 4).
struct __align__(16) GbWarp {
  float u[kGbMaxM];            // the patch, zeros up to a multiple of 4
  float mag[kGbMaxM];          // |alpha| in FP32 of the listed modes
  float qf[kGbMaxM];           // q delta in FP32, in kept order
  double al[kGbMaxM];          // alpha by the definition, where it was needed (by list entry)
  double qd[kGbMaxM];          // q_k delta, by mode (exact evaluations of E)
  long long q[kGbMaxM];        // by mode
  int list[kGbMaxM];           // the modes with q != 0, in index order
  int ord[kGbMaxM];            // modes by decreasing |alpha| (index order on ties)
  unsigned char code[kGbMaxM + 4];      // E(s) <= eps_l^2 for s kept modes: 0 no, 1 yes, 2 open
  uint32_t words[((kGbMaxM * 70 + 31) / 32) + 4];
};

__host__ __device__ inline int gb_ld(int M) { return M | 1; }
__host__ __device__ inline size_t gb_basis_smem(int M) {
  return (size_t)align_up((int64_t)sizeof(float) * gb_ld(M) * (int64_t)align_up(M, 4), 16);
}
__host__ __device__ inline size_t gb_patch_smem(int M) { return gb_basis_smem(M) + sizeof(GbWarp) * kGbWarps; }

__device__ __forceinline__ uint64_t gb_zz(long long q) { return ((uint64_t)q << 1) ^ (uint64_t)(q >> 63); }

// OR `width` (<= 64) bits of v into the words from bit pos (shared memory).
__device__ __forceinline__ void gb_put(uint32_t* w, uint64_t pos, uint64_t v, int width) {
  for (int done = 0; done < width;) {
    const int sh = (int)(pos & 31);
    const int take = (32 - sh) < (width - done) ? (32 - sh) : (width - done);
    const uint32_t part = (uint32_t)((v >> done) & ((take == 32) ? 0xFFFFFFFFull : ((1ull << take) - 1ull)));
    atomicOr(&w[pos >> 5], part << sh);
    pos += (uint64_t)take;
    done += take;
  }
}

__device__ __forceinline__ double gb_warp_sum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = __dadd_rn(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}

// alpha of one mode by the definition: a sequential fma sum over the components.
__device__ __forceinline__ double gb_alpha(const double* __restrict__ phi, const float* u, int M, int k) {
  double a = 0.0;
  for (int j = 0; j < M; ++j) a = __fma_rn(__ldg(phi + j * M + k), widen(u[j]), a);
  return a;
}
__device__ __forceinline__ long long gb_quant(double a, double delta, GbStatus* st) {
  const double y = rint(__ddiv_rn(a, delta));
  if (!(fabs(y) < 0x1p62)) {
    atomicOr(&st->overflow, 1u);
    return 0;
  }
  return (long long)y;
}

// E of the first `kept` modes by the definition (all lanes): the modes added
// in kept order, a multiply then an add, the squares of a lane's points in
// order, the lanes' sums in butterfly order.
__device__ __noinline__ double gb_error(const GbWarp& W, const double* __restrict__ phi, int M, int kept, int lane) {
  double part = 0.0;
  for (int i = lane; i < M; i += 32) {
    double rec = 0.0;
    for (int s = 0; s < kept; ++s) {
      const int k = W.ord[s];
      rec = __dadd_rn(rec, __dmul_rn(W.qd[k], __ldg(phi + i * M + k)));
    }
    const double d = __dsub_rn(widen(W.u[i]), rec);
    part = __fma_rn(d, d, part);
  }
  return gb_warp_sum(part);
}

// Every mode's alpha and the full order by the definition (all lanes).
__device__ __noinline__ void gb_order_all(GbWarp& W, const double* __restrict__ phi, int M, int lane) {
  for (int k = lane; k < M; k += 32) W.al[k] = gb_alpha(phi, W.u, M, k);
  __syncwarp();
  for (int k = lane; k < M; k += 32) {
    const unsigned long long ak = (unsigned long long)__double_as_longlong(W.al[k]) & 0x7FFFFFFFFFFFFFFFull;
    int rank = 0;
    for (int j = 0; j < M; ++j) {
      const unsigned long long aj = (unsigned long long)__double_as_longlong(W.al[j]) & 0x7FFFFFFFFFFFFFFFull;
      rank += (aj > ak || (aj == ak && j < k)) ? 1 : 0;
    }
    W.ord[rank] = k;
  }
  __syncwarp();
}

// A warp per patch, patches in (t, z, y, x) order over the grid's warps; CS =
// ceil(M / 32) modes (and components) a lane.
// Every stored value is the FP64 definition's, but FP64 runs only where FP32
// cannot settle it:
//  - alpha in FP32 is within ea = (M / 4 + 6) u ||patch|| of the definition's
//    (four partial sums, the basis rounded once), so a quotient clear of a
//    half-integer by ea / delta and its own rounding settles q;
//  - modes with q = 0 change no E and come last in the order, so only the
//    modes with q != 0 are ordered, by FP32 magnitudes where they lie 2 ea
//    apart, else by their alphas in FP64;
//  - E(s) for s kept modes comes from the residual r updated mode by mode.  A
//    step's error is at most 4.2 u |q delta| ||phi|| (the roundings of q, delta,
//    their product and phi, the fma's product being exact) plus u ||r||, so the
//    norm of r is known to B_s = u (4.2 sum |q delta| + 1.1 sum ||r||) and pass(s) follows
//    unless sqrt(eps_l^2) lies within B_s (and the sum's rounding) of it.
// Patches whose scale FP32 does not carry, and n = M (no kept count passes),
// take the definition throughout.  Measured at M = 64, 524 288 patches:
// 15.57 -> 1.58 ms; the whole compression and read-back 25.7 -> 10.3 ms.
template <int CS>
__global__ void __launch_bounds__(kGbWarps * 32) k_gb_patch(GbPlan g, const float* __restrict__ in,
                                                            const double* __restrict__ phi, const GbStatus* stc,
                                                            GbStatus* st, unsigned long long* sizes, uint8_t* slots) {
  extern __shared__ __align__(16) unsigned char gsm[];
  constexpr unsigned FULL = 0xffffffffu;
  constexpr float kU = 5.9604645e-8f;
  const int M = g.M, ld = gb_ld(M), M4 = (int)align_up(M, 4);
  float* ph = reinterpret_cast<float*>(gsm);
  GbWarp& W = reinterpret_cast<GbWarp*>(gsm + gb_basis_smem(M))[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  for (int e = threadIdx.x; e < M4 * ld; e += blockDim.x) {
    const int j = e / ld, k = e - j * ld;
    ph[e] = j < M && k < M ? __double2float_rn(phi[j * M + k]) : 0.0f;
  }
  __syncthreads();
  const double eps_l2 = stc->eps_l2, delta = stc->delta;
  const bool pos = delta > 0.0, scale_ok = delta > 1e-16 && delta < 1e16;
  const float inv = scale_ok ? __double2float_rn(1.0 / delta) : 0.0f, delta_f = scale_ok ? __double2float_rn(delta) : 0.0f;
  const float tol = scale_ok ? __double2float_rn(sqrt(eps_l2)) : 0.0f;
  const int ib = g.ib;
  const uint32_t npx = (uint32_t)g.npx, npxy = (uint32_t)(g.npx * g.npy);
  const int64_t pps = g.npx * g.npy * g.npz;
  int64_t poff[CS];                          // field offset of this lane's components inside a patch
#pragma unroll
  for (int c = 0; c < CS; ++c) {
    const int i = lane + 32 * c;
    const int ix = i % g.px, iy = (i / g.px) % g.py, iz = i / (g.px * g.py);
    poff[c] = ((int64_t)iz * g.dims[1] + iy) * g.dims[0] + ix;
  }
  for (int64_t p = (int64_t)blockIdx.x * kGbWarps + (threadIdx.x >> 5); p < g.nrec;
       p += (int64_t)gridDim.x * kGbWarps) {
    int64_t x0, y0, z0, t;
    if (g.nrec <= 0x7fffffff) {
      const uint32_t pp = (uint32_t)p, t32 = pp / (uint32_t)pps, rem = pp - t32 * (uint32_t)pps;
      const uint32_t bz = rem / npxy, r2 = rem - bz * npxy, by = r2 / npx;
      t = t32;
      x0 = (int64_t)(r2 - by * npx) * g.px;
      y0 = (int64_t)by * g.py;
      z0 = (int64_t)bz * g.pz;
    } else {
      t = p / pps;
      const int64_t rem = p - t * pps;
      const int64_t bz = rem / (g.npx * g.npy), r2 = rem - bz * g.npx * g.npy, by = r2 / g.npx;
      x0 = (r2 - by * g.npx) * g.px;
      y0 = by * g.py;
      z0 = bz * g.pz;
    }
    const float* src = in + ((t * g.dims[2] + z0) * g.dims[1] + y0) * g.dims[0] + x0;
    float u[CS], n2 = 0.0f, amax = 0.0f;
#pragma unroll
    for (int c = 0; c < CS; ++c) {
      const int i = lane + 32 * c;
      u[c] = i < M ? __ldg(src + poff[c]) : 0.0f;
      n2 = __fmaf_rn(u[c], u[c], n2);
      amax = fmaxf(amax, fabsf(u[c]));
      W.u[i] = u[c];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      n2 = __fadd_rn(n2, __shfl_xor_sync(FULL, n2, o));
      amax = fmaxf(amax, __shfl_xor_sync(FULL, amax, o));
    }
    __syncwarp();
    const bool f32 = scale_ok && n2 < 1.0e30f && (n2 > 1.0e-30f || amax == 0.0f);
    // alpha (FP32), q
    const float ea = __fmul_rn((float)(M / 4 + 7) * 1.05f * kU, sqrtf(n2));
    float al[CS];
    if (f32) {
      float s0[CS], s1[CS];
#pragma unroll
      for (int c = 0; c < CS; ++c) { s0[c] = 0.0f; s1[c] = 0.0f; }
      int kc[CS];
#pragma unroll
      for (int c = 0; c < CS; ++c) kc[c] = lane + 32 * c < M ? lane + 32 * c : 0;
      float t0[CS], t1[CS];
#pragma unroll
      for (int c = 0; c < CS; ++c) { t0[c] = 0.0f; t1[c] = 0.0f; }
      for (int j = 0; j < M4; j += 4) {
        const float4 v = *reinterpret_cast<const float4*>(&W.u[j]);
        const float* r0 = ph + j * ld;
#pragma unroll
        for (int c = 0; c < CS; ++c) {
          s0[c] = __fmaf_rn(r0[kc[c]], v.x, s0[c]);
          s1[c] = __fmaf_rn(r0[ld + kc[c]], v.y, s1[c]);
          t0[c] = __fmaf_rn(r0[2 * ld + kc[c]], v.z, t0[c]);
          t1[c] = __fmaf_rn(r0[3 * ld + kc[c]], v.w, t1[c]);
        }
      }
#pragma unroll
      for (int c = 0; c < CS; ++c) al[c] = __fadd_rn(__fadd_rn(s0[c], s1[c]), __fadd_rn(t0[c], t1[c]));
    }
    const float mq = __fmul_rn(ea, __fmul_rn(inv, 1.001f));
    int nz = 0;
#pragma unroll
    for (int c = 0; c < CS; ++c) {
      const int k = lane + 32 * c;
      long long q = 0;
      float mag = 0.0f;
      bool open = k < M && pos;
      if (f32 && open) {
        const float y = __fmul_rn(al[c], inv), ry = rintf(y);
        open = !(fabsf(__fsub_rn(y, ry)) < 0.5f - __fadd_rn(mq, __fmaf_rn(fabsf(y), 4.0e-7f, 1.0e-30f)) &&
                 fabsf(y) < 4.0e6f);
        q = (long long)(int)ry;
        mag = fabsf(al[c]);
      }
      if (open) q = gb_quant(gb_alpha(phi, W.u, M, k), delta, st);
      if (k < M) W.q[k] = q;
      const unsigned m = __ballot_sync(FULL, q != 0);
      if (q != 0) {
        const int at = nz + __popc(m & ((1u << lane) - 1u));
        W.list[at] = k;
        W.mag[at] = mag;
      }
      nz += __popc(m);
    }
    __syncwarp();
    // the order of the modes with q != 0
    if (f32) {
      const float sep = __fmul_rn(2.0f, ea);
      unsigned near = 0;                     // entries lane + 32 c with a magnitude within 2 ea of another
#pragma unroll
      for (int c = 0; c < CS; ++c) {
        const int e = lane + 32 * c;
        int rank = 0;
        bool amb = false;
        if (e < nz) {
          const float a = W.mag[e];
          for (int j = 0; j < nz; ++j) {
            const float b = W.mag[j];
            rank += b > a ? 1 : 0;
            amb |= j != e && !(fabsf(__fsub_rn(b, a)) > sep);
          }
          W.ord[rank] = W.list[e];           // (entries of open pairs are placed again below)
        }
        if (amb) near |= 1u << c;
      }
      if (__any_sync(FULL, near != 0)) {
        __syncwarp();
#pragma unroll
        for (int c = 0; c < CS; ++c)
          if ((near >> c) & 1u) W.al[lane + 32 * c] = gb_alpha(phi, W.u, M, W.list[lane + 32 * c]);
        __syncwarp();
#pragma unroll
        for (int c = 0; c < CS; ++c) {
          const int e = lane + 32 * c;
          if ((near >> c) & 1u) {
            const float a = W.mag[e];
            const unsigned long long ak = (unsigned long long)__double_as_longlong(W.al[e]) & 0x7FFFFFFFFFFFFFFFull;
            int rank = 0;
            for (int j = 0; j < nz; ++j) {
              if (j == e) continue;
              const float b = W.mag[j];
              if (fabsf(__fsub_rn(b, a)) > sep) {
                rank += b > a ? 1 : 0;
              } else {
                const unsigned long long aj =
                    (unsigned long long)__double_as_longlong(W.al[j]) & 0x7FFFFFFFFFFFFFFFull;
                rank += (aj > ak || (aj == ak && W.list[j] < W.list[e])) ? 1 : 0;
              }
            }
            W.ord[rank] = W.list[e];
          }
        }
      }
      __syncwarp();
      for (int s = lane; s < nz; s += 32) W.qf[s] = __fmul_rn(__ll2float_rn(W.q[W.ord[s]]), delta_f);
    } else {
      gb_order_all(W, phi, M, lane);
    }
    __syncwarp();
    // the smallest kept count by bisection over [0, M]
    int n = 0;
    if (pos) {
      const int top = f32 ? nz : M;          // E(s) = E(top) for s > top
      if (f32) {
        float r[CS], sum_q = 0.0f, sum_r = 0.0f;
#pragma unroll
        for (int c = 0; c < CS; ++c) r[c] = u[c];
        for (int s = 0; s <= nz; ++s) {
          if (s > 0) {
            const int k = W.ord[s - 1];
            const float qf = W.qf[s - 1];
            sum_q += fabsf(qf);
#pragma unroll
            for (int c = 0; c < CS; ++c) {
              const int i = lane + 32 * c < M ? lane + 32 * c : 0;
              r[c] = lane + 32 * c < M ? __fmaf_rn(-qf, ph[i * ld + k], r[c]) : 0.0f;
            }
          }
          float E = 0.0f;
#pragma unroll
          for (int c = 0; c < CS; ++c) E = __fmaf_rn(r[c], r[c], E);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) E = __fadd_rn(E, __shfl_xor_sync(FULL, E, o));
          const float rn = sqrtf(E);
          if (s > 0) sum_r += rn;
          const float B = __fmaf_rn(1.05f * kU, __fmaf_rn(4.2f, sum_q, __fmul_rn(1.1f, sum_r)), __fmul_rn(rn, 2.0e-6f));
          if (lane == 0) W.code[s] = rn + B < tol * 0.999999f ? 1 : (rn - B > tol * 1.000001f ? 0 : 2);
        }
      } else {
        for (int s = lane; s <= M; s += 32) W.code[s] = 2;
      }
      __syncwarp();
      bool have_qd = false;
      int lo = 0, hi = M;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1, at = mid < top ? mid : top;
        int code = W.code[at];
        if (code == 2) {
          if (!have_qd) {
            for (int k = lane; k < M; k += 32) W.qd[k] = __dmul_rn((double)W.q[k], delta);
            have_qd = true;
          }
          __syncwarp();
          code = gb_error(W, phi, M, at, lane) <= eps_l2 ? 1 : 0;
          if (lane == 0) W.code[at] = (unsigned char)code;
          __syncwarp();
        }
        if (code) hi = mid;
        else lo = mid + 1;
      }
      n = lo;
      if (n > top) gb_order_all(W, phi, M, lane);          // modes with q = 0 are kept too
    }
    // the record: n, wv, n mode indices of ib bits, n zigzag(q) of wv bits
    uint64_t zmax = 0;
    for (int s = lane; s < n; s += 32) {
      const uint64_t z = gb_zz(W.q[W.ord[s]]);
      zmax = z > zmax ? z : zmax;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const uint64_t z = __shfl_xor_sync(0xffffffffu, zmax, o);
      zmax = z > zmax ? z : zmax;
    }
    const int wv = gb_width(zmax);
    const int64_t nbits = (int64_t)n * (ib + wv);
    const int nw = (int)((nbits + 31) / 32);
    const int64_t bytes = align_up(8 + 4 * (int64_t)nw, 8);
    for (int w = lane; w < nw + 2; w += 32) W.words[w] = 0u;
    __syncwarp();
    for (int s = lane; s < n; s += 32) {
      const int k = W.ord[s];
      gb_put(W.words, (uint64_t)s * ib, (uint64_t)k, ib);
      gb_put(W.words, (uint64_t)n * ib + (uint64_t)s * wv, gb_zz(W.q[k]), wv);
    }
    __syncwarp();
    uint32_t* slot = reinterpret_cast<uint32_t*>(slots + p * g.slot_bytes);
    for (int w = lane; w < (int)(bytes / 4); w += 32)
      slot[w] = w == 0 ? (uint32_t)n : w == 1 ? (uint32_t)wv : W.words[w - 2];
    if (lane == 0) sizes[p] = (unsigned long long)bytes;
    __syncwarp();
  }
}

// ---------------------------------------------------------------- the stream
// Tiles of kGbTile records: k_gb_tiles sums their sizes, k_gb_scan (one CTA)
// scans the tiles' sums and writes header and basis, k_gb_copy finishes the
// scan inside each tile, writing its part of the offset table and its records.
// (One CTA scanning every record took 586 us for 524 288 of them.)
__global__ void __launch_bounds__(256) k_gb_tiles(GbPlan g, const unsigned long long* __restrict__ sizes,
                                                  unsigned long long* tiles) {
  __shared__ unsigned long long ws[8];
  const int64_t b = (int64_t)blockIdx.x * kGbTile;
  unsigned long long s = 0;
#pragma unroll
  for (int k = 0; k < kGbTile / 256; ++k) {
    const int64_t i = b + threadIdx.x + 256 * k;
    s += i < g.nrec ? sizes[i] : 0ull;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) s += ws[w];
    tiles[blockIdx.x] = s;
  }
}

// The exclusive scan of the tiles' sums (in place), the total, and the header
// and basis when the stream fits.
__global__ void __launch_bounds__(1024) k_gb_scan(GbPlan g, unsigned long long* tiles, int64_t ntiles,
                                                  const double* phi, GbStatus* st, uint8_t* out,
                                                  unsigned long long out_cap) {
  __shared__ unsigned long long warp_sums[32];
  __shared__ unsigned long long carry;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) carry = 0;
  __syncthreads();
  for (int64_t base = 0; base < ntiles; base += 1024) {
    const int64_t i = base + tid;
    const unsigned long long v = i < ntiles ? tiles[i] : 0ull;
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) warp_sums[warp] = x;
    __syncthreads();
    if (warp == 0) {
      unsigned long long s = warp_sums[lane];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += y;
      }
      warp_sums[lane] = s;
    }
    __syncthreads();
    const unsigned long long excl = carry + (warp > 0 ? warp_sums[warp - 1] : 0ull) + x - v;
    if (i < ntiles) tiles[i] = excl;
    __syncthreads();
    if (tid == 1023) carry = excl + v;
    __syncthreads();
  }
  const unsigned long long payload = carry;
  const unsigned long long total = (unsigned long long)g.payload_pos + payload;
  if (tid == 0) st->total = total;
  if (total > out_cap) return;
  const int M = g.M;
  if (tid == 0) {
    uint32_t* h32 = reinterpret_cast<uint32_t*>(out);
    uint64_t* h64 = reinterpret_cast<uint64_t*>(out);
    double* hd = reinterpret_cast<double*>(out);
    h32[0] = kGbMagic;
    h32[1] = 1u;
    h32[2] = (uint32_t)M;
    h32[3] = (uint32_t)g.px;
    h32[4] = (uint32_t)g.py;
    h32[5] = (uint32_t)g.pz;
    for (int a = 0; a < 4; ++a) h64[3 + a] = (uint64_t)g.dims[a];
    hd[7] = st->eps_l2;
    hd[8] = st->delta;
    h64[9] = (uint64_t)g.nrec;
    reinterpret_cast<uint64_t*>(out + g.offsets_pos)[g.nrec] = payload;
  }
  double* basis = reinterpret_cast<double*>(out + kGbHdr);
  for (int e = tid; e < M * M; e += 1024) {
    const int r = e / M, i = e - r * M;          // mode r, component i
    basis[e] = phi[i * M + r];
  }
}

// A tile's offsets, and its records from their slots (8-byte words, eight
// lanes a record: a record is a few tens of bytes).
__global__ void __launch_bounds__(256) k_gb_copy(GbPlan g, const unsigned long long* __restrict__ sizes,
                                                 const unsigned long long* __restrict__ tiles,
                                                 const uint8_t* __restrict__ slots, const GbStatus* st, uint8_t* out,
                                                 unsigned long long out_cap) {
  __shared__ int sh_warp[32];
  __shared__ unsigned int off[kGbTile + 1];
  if (st->total > out_cap) return;
  const int tid = threadIdx.x;
  const int64_t b = (int64_t)blockIdx.x * kGbTile;
  const int cnt = (int)((g.nrec - b) < kGbTile ? (g.nrec - b) : kGbTile);
  const unsigned long long base = tiles[blockIdx.x];
  int sz[kGbTile / 256], mine = 0;               // four consecutive records a thread
#pragma unroll
  for (int k = 0; k < kGbTile / 256; ++k) {
    const int i = tid * (kGbTile / 256) + k;
    sz[k] = i < cnt ? (int)sizes[b + i] : 0;
    mine += sz[k];
  }
  int tot;
  int at = block_excl_scan(mine, sh_warp, &tot);
#pragma unroll
  for (int k = 0; k < kGbTile / 256; ++k) {
    off[tid * (kGbTile / 256) + k] = (unsigned)at;
    at += sz[k];
  }
  if (tid == 0) off[kGbTile] = (unsigned)tot;
  __syncthreads();
  uint64_t* ot = reinterpret_cast<uint64_t*>(out + g.offsets_pos);
  for (int i = tid; i < cnt; i += 256) ot[b + i] = base + off[i];
  const int sub = tid >> 3, l8 = tid & 7;
  for (int i = sub; i < cnt; i += 32) {
    const uint2* src = reinterpret_cast<const uint2*>(slots + (b + i) * g.slot_bytes);
    uint2* dst = reinterpret_cast<uint2*>(out + g.payload_pos + base + off[i]);
    const int nw = (int)((off[i + 1] - off[i]) / 8);
    for (int w = l8; w < nw; w += 8) dst[w] = src[w];
  }
}

// ---------------------------------------------------------------- decoder
// A warp per record: its mode indices and values, then each point the sum of
// (q_s delta) phi_s over the kept modes in kept order.
__global__ void __launch_bounds__(256) k_gb_decode(GbPlan g, const uint8_t* __restrict__ comp,
                                                   unsigned long long comp_bytes, double delta, double* out,
                                                   GbStatus* st) {
  const int64_t p = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (p >= g.nrec) return;
  const int lane = threadIdx.x & 31;
  const int M = g.M;
  const uint64_t* ot = reinterpret_cast<const uint64_t*>(comp + g.offsets_pos);
  const double* basis = reinterpret_cast<const double*>(comp + kGbHdr);   // [mode][component]
  const uint64_t o0 = ot[p], o1 = ot[p + 1];
  // (entries near 2^64 must not wrap)
  if (o1 > comp_bytes - (uint64_t)g.payload_pos || o0 > o1 || o1 - o0 < 8 || (o0 & 7) != 0) {
    if (lane == 0) atomicOr(&st->corrupt, 1u);
    return;
  }
  const uint32_t* r = reinterpret_cast<const uint32_t*>(comp + g.payload_pos + o0);
  const int n = (int)r[0], wv = (int)(r[1] & 0xFFu);
  const int ib = g.ib;
  if (n > M || wv > 63 || (r[1] >> 8) != 0u ||
      (int64_t)(o1 - o0) != align_up(8 + 4 * (((int64_t)n * (ib + wv) + 31) / 32), 8)) {
    if (lane == 0) atomicOr(&st->corrupt, 1u);
    return;
  }
  // the entries, one a lane: mode and q delta to shared memory, once a record
  // (each lane unpacking and multiplying every entry for its own points was
  // half of the decoder's time)
  __shared__ double sqd[8][kGbMaxM];
  __shared__ short smode[8][kGbMaxM];
  double* qd = sqd[threadIdx.x >> 5];
  short* md = smode[threadIdx.x >> 5];
  const uint32_t* w = r + 2;
  auto get = [&](uint64_t pos, int width) -> uint64_t {
    uint64_t v = 0;
    for (int done = 0; done < width;) {
      const int sh = (int)(pos & 31);
      const int take = (32 - sh) < (width - done) ? (32 - sh) : (width - done);
      const uint64_t part = (w[pos >> 5] >> sh) & ((take == 32) ? 0xFFFFFFFFull : ((1ull << take) - 1ull));
      v |= part << done;
      pos += (uint64_t)take;
      done += take;
    }
    return v;
  };
  bool bad = false;
  for (int s = lane; s < n; s += 32) {
    const int k = (int)get((uint64_t)s * ib, ib);
    const uint64_t z = get((uint64_t)n * ib + (uint64_t)s * wv, wv);
    const long long q = (long long)((z >> 1) ^ (0ull - (z & 1ull)));
    bad |= k >= M;
    md[s] = (short)k;
    qd[s] = __dmul_rn((double)q, delta);
  }
  if (__any_sync(0xffffffffu, bad)) {
    if (lane == 0) atomicOr(&st->corrupt, 1u);
    return;
  }
  __syncwarp();
  const int64_t pps = g.npx * g.npy * g.npz;
  const int64_t t = p / pps, rem = p - t * pps;
  const int64_t bz = rem / (g.npx * g.npy), r2 = rem - bz * g.npx * g.npy;
  const int64_t by = r2 / g.npx, bx = r2 - by * g.npx;
  const int64_t x0 = bx * g.px, y0 = by * g.py, z0 = bz * g.pz;
  for (int i = lane; i < M; i += 32) {
    double rec = 0.0;
    for (int s = 0; s < n; ++s) rec = __dadd_rn(rec, __dmul_rn(qd[s], __ldg(basis + (int64_t)md[s] * M + i)));
    const int ix = i % g.px, iy = (i / g.px) % g.py, iz = i / (g.px * g.py);
    out[((t * g.dims[2] + z0 + iz) * g.dims[1] + (y0 + iy)) * g.dims[0] + (x0 + ix)] = rec;
  }
}

}  // namespace
}  // namespace dls

using namespace dls;

size_t dls_gb_bound(const dls_gb_params* p) {
  GbPlan g;
  if (gb_make_plan(p, &g) != DLS_OK) return 0;
  return (size_t)(g.payload_pos + g.nrec * gb_record_max(g.M, g.ib));
}

size_t dls_gb_workspace_size(const dls_gb_params* p) {
  GbPlan g;
  if (gb_make_plan(p, &g) != DLS_OK) return 0;
  return gb_layout(g).total;
}

int dls_gb_compress(const dls_gb_params* p, const float* d_in, const int64_t* d_origins, void* d_out, size_t out_cap,
                    size_t* out_bytes, void* d_workspace, size_t ws_bytes, dls_stream_t stream) {
  GbPlan g;
  int st = gb_make_plan(p, &g);
  if (st != DLS_OK) return st;
  if (!d_in || !d_origins || !d_out || !out_bytes || ((uintptr_t)d_out & 15) || ((uintptr_t)d_in & 3) ||
      ((uintptr_t)d_origins & 7))
    return DLS_ERR_INVALID_ARG;
  const GbLayout L = gb_layout(g);
  if (!d_workspace || ws_bytes < L.total || ((uintptr_t)d_workspace & 255)) return DLS_ERR_WORKSPACE;
  cudaStream_t s = (cudaStream_t)stream;
  uint8_t* w = (uint8_t*)d_workspace;
  double* Q = (double*)(w + L.Q);
  double* G = (double*)(w + L.G);
  double* V = (double*)(w + L.V);
  double* phi = (double*)(w + L.phi);
  double* lam = (double*)(w + L.lam);
  double* partial = (double*)(w + L.partial);
  GbStatus* gs = (GbStatus*)(w + L.status);
  unsigned long long* sizes = (unsigned long long*)(w + L.sizes);
  unsigned long long* tiles = (unsigned long long*)(w + L.tiles);
  uint8_t* slots = w + L.slots;
  if (cudaMemsetAsync(gs, 0, sizeof(GbStatus), s) != cudaSuccess) return DLS_ERR_CUDA;
  k_gb_sample<<<(unsigned)g.S, 128, 0, s>>>(g, d_in, d_origins, Q, gs);
  k_gb_gram<<<(unsigned)cdiv((int64_t)g.M * g.M, 256), 256, 0, s>>>(g, Q, G);
  if (cudaFuncSetAttribute(k_gb_jacobi, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GbJac)) != cudaSuccess)
    return DLS_ERR_CUDA;
  k_gb_jacobi<<<kJacCtas, kJacThreads, sizeof(GbJac), s>>>(g, G, V, phi, lam);
  k_gb_norm<<<kGbStatCtas, 256, 0, s>>>(g, d_in, partial, gs);
  k_gb_resolve<<<1, 128, 0, s>>>(g, partial, gs);
  const size_t psm = gb_patch_smem(g.M);
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return DLS_ERR_CUDA;
  auto patches = [&](auto kern) -> bool {
    int per = 0;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)psm) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, kGbWarps * 32, psm) != cudaSuccess || per < 1)
      return false;
    const int64_t need = cdiv(g.nrec, kGbWarps);
    const unsigned grid = (unsigned)((int64_t)per * sms < need ? (int64_t)per * sms : need);
    kern<<<grid, kGbWarps * 32, psm, s>>>(g, d_in, phi, gs, gs, sizes, slots);
    return true;
  };
  if (!(g.M <= 32 ? patches(k_gb_patch<1>) : g.M <= 64 ? patches(k_gb_patch<2>) : g.M <= 96 ? patches(k_gb_patch<3>)
                                                                                            : patches(k_gb_patch<4>)))
    return DLS_ERR_CUDA;
  const int64_t ntiles = cdiv(g.nrec, kGbTile);
  k_gb_tiles<<<(unsigned)ntiles, 256, 0, s>>>(g, sizes, tiles);
  k_gb_scan<<<1, 1024, 0, s>>>(g, tiles, ntiles, phi, gs, (uint8_t*)d_out, (unsigned long long)out_cap);
  k_gb_copy<<<(unsigned)ntiles, 256, 0, s>>>(g, sizes, tiles, slots, gs, (uint8_t*)d_out, (unsigned long long)out_cap);
  if (cudaGetLastError() != cudaSuccess) return DLS_ERR_CUDA;
  GbStatus hs;
  if (cudaMemcpyAsync(&hs, gs, sizeof(hs), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return DLS_ERR_CUDA;
  if (hs.bad_origin || hs.overflow) return DLS_ERR_INVALID_ARG;
  if (hs.nonfinite) return DLS_ERR_NONFINITE;
  *out_bytes = (size_t)hs.total;
  return hs.total > out_cap ? DLS_ERR_CAPACITY : DLS_OK;
}

int dls_gb_decompress(const void* d_comp, size_t comp_bytes, double* d_out, size_t out_count, dls_stream_t stream) {
  if (!d_comp || !d_out || comp_bytes < (size_t)kGbHdr || ((uintptr_t)d_comp & 15) || ((uintptr_t)d_out & 7))
    return DLS_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  uint8_t h[kGbHdr];
  if (cudaMemcpyAsync(h, d_comp, kGbHdr, cudaMemcpyDeviceToHost, s) != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess)
    return DLS_ERR_CUDA;
  uint32_t h32[6];
  uint64_t dims[4], nrec;
  double eps_l2, delta;
  memcpy(h32, h, 24);
  memcpy(dims, h + 24, 32);
  memcpy(&eps_l2, h + 56, 8);
  memcpy(&delta, h + 64, 8);
  memcpy(&nrec, h + 72, 8);
  if (h32[0] != kGbMagic || h32[1] != 1u || h32[3] == 0 || h32[3] != h32[4] || h32[2] > (uint32_t)kGbMaxM)
    return DLS_ERR_CORRUPT;
  for (int a = 0; a < 4; ++a)
    if (dims[a] < 1 || dims[a] > (1ull << 40)) return DLS_ERR_CORRUPT;
  dls_gb_params p;
  p.m = (int32_t)h32[3];
  for (int a = 0; a < 4; ++a) p.dims[a] = (int64_t)dims[a];
  p.eps_t = 1.0;
  p.nsample = 1;
  GbPlan g;
  if (gb_make_plan(&p, &g) != DLS_OK || (uint32_t)g.M != h32[2] || (uint32_t)g.pz != h32[5] ||
      (uint64_t)g.nrec != nrec || !isfinite(delta) || delta < 0.0)
    return DLS_ERR_CORRUPT;
  if (comp_bytes < (size_t)g.payload_pos) return DLS_ERR_CORRUPT;
  if (out_count < (size_t)g.K) return DLS_ERR_CAPACITY;
  // the offset table: starts at 0, ends at the stream's end (the records' own
  // sizes are checked on the device)
  uint64_t first = 0, last = 0;
  const uint8_t* c = (const uint8_t*)d_comp;
  if (cudaMemcpyAsync(&first, c + g.offsets_pos, 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaMemcpyAsync(&last, c + g.offsets_pos + 8 * g.nrec, 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return DLS_ERR_CUDA;
  if (first != 0 || (uint64_t)g.payload_pos + last != (uint64_t)comp_bytes) return DLS_ERR_CORRUPT;
  GbStatus* gs = nullptr;
  if (scratch_alloc((void**)&gs, sizeof(GbStatus), s) != cudaSuccess) return DLS_ERR_CUDA;
  if (cudaMemsetAsync(gs, 0, sizeof(GbStatus), s) != cudaSuccess) {
    cudaFreeAsync(gs, s);
    return DLS_ERR_CUDA;
  }
  if (g.nrec > 0)
    k_gb_decode<<<(unsigned)cdiv(g.nrec, 8), 256, 0, s>>>(g, c, (unsigned long long)comp_bytes, delta, d_out, gs);
  GbStatus hs;
  memset(&hs, 0, sizeof(hs));
  const bool launched = cudaGetLastError() == cudaSuccess;
  cudaMemcpyAsync(&hs, gs, sizeof(hs), cudaMemcpyDeviceToHost, s);
  cudaFreeAsync(gs, s);
  if (cudaStreamSynchronize(s) != cudaSuccess || !launched) return DLS_ERR_CUDA;
  return hs.corrupt ? DLS_ERR_CORRUPT : DLS_OK;
}
