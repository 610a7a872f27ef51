// Decompression (Sec. 2.6 and Algorithm 2 of arXiv 2601.20113) and
// verification (Sec. 2.4 metrics).
//
// Decode contract: for every point, acc = 0; for k = 0..r-1,
// acc = fma(chat[l][k], Vst[j][k], acc) in the field dtype, with
// chat = dtype(q) * dtype(delta).  Then xtilde = fma(dtype(k), dtype(2eb), acc)
// where the correction k is nonzero, and escaped points take their raw value.
// Every structural field of a record is validated against the geometry before
// use.  k_decode_f32 takes float32 plans of time-side blocks of up to 16 time
// steps and 65 536 points (persistent CTAs, a record brought in by one bulk
// copy), k_decode the others, a CTA a block.
#include "dls_internal.cuh"

namespace dls {
namespace {

constexpr int kDecThreads = 256;
// Shared-memory words for a record's coefficient and correction sections
// (72 KB: three CTAs per SM, as the launch bounds ask of the registers).
constexpr int kDecStageWords = 18432;

// Whether a record's table entries lie in order inside the payload (`room` bytes
// after payload_pos), the first a multiple of 16: entries near 2^64 must not wrap.
__device__ __forceinline__ bool record_in(uint64_t o0, uint64_t o1, uint64_t room) {
  return o1 <= room && o0 <= o1 && o1 - o0 >= 16 && (o0 & 15) == 0;
}

template <typename T> __device__ __forceinline__ T dq(int32_t q, T d);
template <> __device__ __forceinline__ float dq<float>(int32_t q, float d) { return __fmul_rn(__int2float_rn(q), d); }
template <> __device__ __forceinline__ double dq<double>(int32_t q, double d) { return __dmul_rn((double)q, d); }
template <typename T> __device__ __forceinline__ T tf(T a, T b, T c);
template <> __device__ __forceinline__ float tf<float>(float a, float b, float c) { return __fmaf_rn(a, b, c); }
template <> __device__ __forceinline__ double tf<double>(double a, double b, double c) { return __fma_rn(a, b, c); }
template <typename T> __device__ __forceinline__ T from_d(double x);
template <> __device__ __forceinline__ float from_d<float>(double x) { return __double2float_rn(x); }
template <> __device__ __forceinline__ double from_d<double>(double x) { return x; }

__device__ __forceinline__ uint32_t get_bits(const uint32_t* w, uint64_t pos, int width) {
  if (width == 0) return 0;
  const uint64_t wi = pos >> 5;
  const int sh = (int)(pos & 31);
  uint64_t v = w[wi] >> sh;
  if (sh + width > 32) v |= (uint64_t)w[wi + 1] << (32 - sh);
  return (uint32_t)(v & (width == 32 ? 0xffffffffull : ((1ull << width) - 1)));
}

// get_bits for bit positions below 2^32 (a column of L <= 2^26 values of at
// most 32 bits); width 0 reads nothing.
__device__ __forceinline__ uint32_t get_bits32(const uint32_t* w, uint32_t pos, int width) {
  if (width == 0) return 0;
  const uint32_t wi = pos >> 5;
  const int sh = (int)(pos & 31);
  uint32_t v = w[wi] >> sh;
  if (sh + width > 32) v |= w[wi + 1] << (32 - sh);
  return width == 32 ? v : (v & ((1u << width) - 1u));
}

template <int V> struct RankC { static constexpr int value = V; };
template <bool V> struct BoolC { static constexpr bool value = V; };

// Field offset of a block's spatial point ls (x fastest) without the time
// step: 32-bit division (a block's extents are small), once per point.
__device__ __forceinline__ int64_t spatial_off(const Plan& p, const Geom& g, int ls) {
  const int sx = g.sx, sxy = g.sx * g.sy;
  const int lz = ls / sxy, rxy = ls - lz * sxy;
  const int ly = rxy / sx, lx = rxy - ly * sx;
  return (int64_t)g.v * p.K + (g.z0 + lz) * (p.dims[0] * p.dims[1]) + (g.y0 + ly) * p.dims[0] + (g.x0 + lx);
}
// elem_index (block element e = t_local * M + s_local) the same way.
__device__ __forceinline__ int64_t elem_off(const Plan& p, const Geom& g, int64_t e) {
  const int64_t lt = e / g.M;
  return spatial_off(p, g, (int)(e - lt * g.M)) + (g.t0 + lt) * p.P;
}

// One block of any shape, rank and correction width, by all NT threads of a
// CTA; stage_sm holds stage_words words.  T16: with the unrolled rows of order 16.
template <typename T, int NM, int NT, bool T16 = false>
__device__ __forceinline__ void decode_block(const Plan& P, const uint8_t* __restrict__ comp, unsigned long long comp_bytes,
                             T* __restrict__ out, Status* st, int64_t bi, uint32_t* stage_sm, int stage_words) {
  __shared__ T vst[NM * NM];
  __shared__ int64_t wbase[NM + 1];
  __shared__ int64_t soff_col[NM];   // spatial-side blocks: field offset of column j (time 0)
  __shared__ int bad;
  const int tid = threadIdx.x;
  const Geom g = block_geom(P, P.b0 + bi);
  const int64_t N = g.N, L = g.L;
  const int n = g.n;
  const int es = (int)sizeof(T);
  const uint64_t* offs = reinterpret_cast<const uint64_t*>(comp + P.offsets_pos);
  const uint64_t o0 = offs[bi], o1 = offs[bi + 1];
  if (!record_in(o0, o1, comp_bytes - (uint64_t)P.payload_pos)) {
    if (tid == 0) atomicOr(&st->corrupt, 1u);
    return;
  }
  const uint8_t* rec = comp + P.payload_pos + o0;
  const uint32_t* rec32 = reinterpret_cast<const uint32_t*>(rec);
  const int r = rec[0], flags = rec[1], wk = rec[2], ib = rec[3];
  const int64_t ncorr = rec32[1], nesc = rec32[2], nbytes = rec32[3];
  // a flag outside raw / spatial side / dense / Rice-coded corrections is refused
  if (nbytes != (int64_t)(o1 - o0) || nbytes < 16 ||
      (flags & ~(int)(kFlagRaw | kFlagSpatial | kFlagDense | kFlagRice)) != 0) {
    if (tid == 0) atomicOr(&st->corrupt, 1u);
    return;
  }
  if (flags & kFlagRaw) {
    if (16 + N * es > nbytes) {
      if (tid == 0) atomicOr(&st->corrupt, 1u);
      return;
    }
    const T* vals = reinterpret_cast<const T*>(rec + 16);
    for (int64_t e = tid; e < N; e += NT) out[elem_off(P, g, e)] = vals[e];
    return;
  }
  const int rcap = P.rank_cap < n ? P.rank_cap : n;
  const uint8_t* wq = rec + 16;
  if (tid == 0) {
    bad = 0;
    if (16 + align_up(r, 8) > nbytes || r > rcap || wk > 32 || ib != bit_width((uint32_t)(N - 1)) || ncorr > N || nesc > N ||
        (((flags & kFlagSpatial) ? 1 : 0) != g.side))
      bad = 1;
    int64_t acc = 0;
    for (int c = 0; c < r && !bad; ++c) {
      if (wq[c] > 32) bad = 1;
      wbase[c] = acc;
      acc += (L * wq[c] + 31) / 32;
    }
    wbase[r] = acc;
    if (!bad) {
      RecLayout lay = rec_layout(r, n, L, N, es, wq, wk, ib, ncorr, nesc);
      if (flags & kFlagRice) {
        // [coded words, kr | wv << 8, chunk bit offsets, coded words]
        if (wk == 0 || (flags & kFlagDense) || lay.off_c + 8 > nbytes) {
          bad = 1;
        } else {
          const uint32_t* cw = reinterpret_cast<const uint32_t*>(rec + lay.off_c);
          if ((cw[1] >> 16) != 0u || (int)(cw[1] & 0xFFu) > kRiceMaxKr || (int)((cw[1] >> 8) & 0xFFu) > 32 ||
              (int64_t)cw[0] > nbytes)
            bad = 1;
          else
            lay = rice_layout(lay, N, cw[0], nesc, es);
        }
        if (!bad && lay.size != nbytes) bad = 1;
      } else if (lay.size != nbytes || (lay.dense ? 1 : 0) != ((flags & kFlagDense) ? 1 : 0)) {
        bad = 1;
      }
    }
  }
  __syncthreads();
  if (bad) {
    if (tid == 0) atomicOr(&st->corrupt, 1u);
    return;
  }
  const bool rice = (flags & kFlagRice) != 0;
  RecLayout lay = rec_layout(r, n, L, N, es, wq, wk, ib, ncorr, nesc);
  if (rice) lay = rice_layout(lay, N, reinterpret_cast<const uint32_t*>(rec + lay.off_c)[0], nesc, es);
  const int v = g.v;
  const double delta = reinterpret_cast<const double*>(comp + kHdr + kVarRec * v)[2];
  const double step = reinterpret_cast<const double*>(comp + kHdr + kVarRec * v)[3];
  const T delta_t = from_d<T>(delta), step_t = from_d<T>(step);
  const T* vin = reinterpret_cast<const T*>(rec + lay.off_v);
  for (int i = tid; i < n * r; i += NT) {
    const int c = i / n, j = i - c * n;
    vst[j * NM + c] = vin[i];
  }
  if (g.side == 1 && tid < n) soff_col[tid] = spatial_off(P, g, tid);
  // the coefficient and correction sections (contiguous words from off_q) go
  // to shared memory in one pass with every load in flight, when they fit;
  // the row loop then reads them at shared-memory latency
  const int64_t cw_at = (lay.off_c - lay.off_q) / 4;
  const int64_t nstage = cw_at + lay.corr_words;
  const bool staged = nstage <= stage_words;
  const uint32_t* qw = reinterpret_cast<const uint32_t*>(rec + lay.off_q);
  if (staged)
    for (int64_t i = tid; i < nstage; i += NT) stage_sm[i] = qw[i];
  __syncthreads();
  if (staged) qw = stage_sm;
  const uint32_t* cw = qw + cw_at;
  const bool dense = lay.dense && wk > 0;
  // Rank 1-8 (the common case) with the rank fixed at compile time: the
  // coefficients of a row in registers, each output r FMAs; the time-side
  // outputs of a row one time plane apart.  Other ranks: guarded up to NM.
  auto rows_fixed = [&](auto RK) {
    constexpr int R = decltype(RK)::value;
    int wqc[R];
    const uint32_t* qc[R];
#pragma unroll
    for (int c = 0; c < R; ++c) { wqc[c] = wq[c]; qc[c] = qw + wbase[c]; }
    for (int64_t l = tid; l < L; l += NT) {
      const int64_t row_off = g.side == 0 ? spatial_off(P, g, (int)l) + g.t0 * P.P : (g.t0 + l) * P.P;
      T ch[R];
#pragma unroll
      for (int c = 0; c < R; ++c) ch[c] = dq<T>(unzigzag(get_bits32(qc[c], (uint32_t)l * (uint32_t)wqc[c], wqc[c])), delta_t);
      T* o = out + row_off;
#pragma unroll 1
      for (int j = 0; j < n; ++j) {
        T acc = T(0);
#pragma unroll
        for (int c = 0; c < R; ++c) acc = tf<T>(ch[c], vst[j * NM + c], acc);
        if (dense) {
          const int32_t kv = unzigzag(get_bits(cw, (uint64_t)a_elem(g, l, j) * wk, wk));
          if (kv != 0) acc = tf<T>((T)kv, step_t, acc);
        }
        if (g.side == 0) {
          *o = acc;
          o += P.P;
        } else {
          out[row_off + soff_col[j]] = acc;
        }
      }
    }
  };
  // float32 time-side blocks of order 16 at ranks 1-4: the 16 outputs of a row
  // unrolled, dense corrections read with 32-bit bit positions one time plane
  // (M wk bits) apart, blocks without them compiled without their test.  (2 GiB
  // in blocks of 32 x 32 x 16 x 16 at 1e-2: 1837 us with the loop above, 1579
  // so; float64 the same either way.)
  auto rows_t16 = [&](auto RK, auto DK) {
    constexpr int R = decltype(RK)::value;
    constexpr bool D = decltype(DK)::value;
    int wqc[R];
    const uint32_t* qc[R];
#pragma unroll
    for (int c = 0; c < R; ++c) { wqc[c] = wq[c]; qc[c] = qw + wbase[c]; }
    const uint32_t pstep = (uint32_t)g.M * (uint32_t)wk;
    for (int l = tid; l < (int)L; l += NT) {
      T ch[R];
#pragma unroll
      for (int c = 0; c < R; ++c) ch[c] = dq<T>(unzigzag(get_bits32(qc[c], (uint32_t)l * (uint32_t)wqc[c], wqc[c])), delta_t);
      T* o = out + spatial_off(P, g, l) + g.t0 * P.P;
      uint32_t pos = (uint32_t)l * (uint32_t)wk;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        T acc = T(0);
#pragma unroll
        for (int c = 0; c < R; ++c) acc = tf<T>(ch[c], vst[j * NM + c], acc);
        if (D) {
          const int32_t kv = unzigzag(get_bits32(cw, pos, wk));
          pos += pstep;
          if (kv != 0) acc = tf<T>((T)kv, step_t, acc);
        }
        *o = acc;
        o += P.P;
      }
    }
  };
  auto rows_t16_d = [&](auto RK) {
    if (dense) rows_t16(RK, BoolC<true>());
    else rows_t16(RK, BoolC<false>());
  };
  if (T16 && g.side == 0 && n == 16 && r >= 1 && r <= 4 && (uint64_t)N * (uint64_t)wk < (1ull << 32)) {
    switch (r) {
      case 1: rows_t16_d(RankC<1>()); break;
      case 2: rows_t16_d(RankC<2>()); break;
      case 3: rows_t16_d(RankC<3>()); break;
      default: rows_t16_d(RankC<4>()); break;
    }
  } else switch (r) {
    case 1: rows_fixed(RankC<1>()); break;
    case 2: rows_fixed(RankC<2>()); break;
    case 3: rows_fixed(RankC<3>()); break;
    case 4: rows_fixed(RankC<4>()); break;
    case 5: rows_fixed(RankC<5>()); break;
    case 6: rows_fixed(RankC<6>()); break;
    case 7: rows_fixed(RankC<7>()); break;
    case 8: rows_fixed(RankC<8>()); break;
    default:
      for (int64_t l = tid; l < L; l += NT) {
        // row l's field offset: a spatial point (time side) or a time step (spatial side)
        const int64_t row_off = g.side == 0 ? spatial_off(P, g, (int)l) + g.t0 * P.P : (g.t0 + l) * P.P;
        T ch[NM];
#pragma unroll
        for (int c = 0; c < NM; ++c) {
          if (c < r) {
            const uint32_t z = get_bits(qw + wbase[c], (uint64_t)l * wq[c], wq[c]);
            ch[c] = dq<T>(unzigzag(z), delta_t);
          } else {
            ch[c] = T(0);
          }
        }
        // one output at a time: unrolled over j, the basis (loop-invariant over
        // rows) would be held in registers, a CTA per SM
#pragma unroll 1
        for (int j = 0; j < n; ++j) {
          {
            T acc = T(0);
#pragma unroll
            for (int c = 0; c < NM; ++c)
              if (c < r) acc = tf<T>(ch[c], vst[j * NM + c], acc);
            const int64_t e = a_elem(g, l, j);
            if (dense) {
              const int32_t kv = unzigzag(get_bits(cw, (uint64_t)e * wk, wk));
              if (kv != 0) acc = tf<T>((T)kv, step_t, acc);
            }
            out[row_off + (g.side == 0 ? (int64_t)j * P.P : soff_col[j])] = acc;
          }
        }
      }
      break;
  }
  __syncthreads();
  if (rice) {
    // chunk by chunk, one thread each: a Rice code gives the zeros before
    // the next nonzero (or the chunk's end), then wv bits give zigzag(k) - 1
    const int kr = (int)(cw[1] & 0xFFu), wv = (int)((cw[1] >> 8) & 0xFFu);
    const int64_t nch = cdiv(N, kRiceChunk);
    const uint32_t* rw = cw + 2 + nch;
    const uint64_t nbits = (uint64_t)cw[0] * 32;
    for (int64_t ch = tid; ch < nch; ch += NT) {
      const int64_t c1 = (ch + 1) * kRiceChunk < N ? (ch + 1) * kRiceChunk : N;
      int64_t e = ch * kRiceChunk;
      uint64_t pos = cw[2 + ch];
      bool ok = true;
      int64_t pg[8];
      int32_t pk[8];
      int npend = 0;
      auto flush = [&]() {
        T val[8];
#pragma unroll
        for (int b = 0; b < 8; ++b) val[b] = b < npend ? out[pg[b]] : T(0);
#pragma unroll
        for (int b = 0; b < 8; ++b)
          if (b < npend) out[pg[b]] = tf<T>((T)pk[b], step_t, val[b]);
        npend = 0;
      };
      for (;;) {
        // the unary part: ones up to a zero
        uint64_t q = 0;
        for (;;) {
          if (pos >= nbits) { ok = false; break; }
          const int avail = (nbits - pos) < 32 ? (int)(nbits - pos) : 32;
          const uint32_t w = get_bits(rw, pos, avail);
          const int t = (~w == 0u) ? 32 : __ffs(~w) - 1;
          if (t >= avail) {
            q += (uint64_t)avail;
            pos += (uint64_t)avail;
            if (q > (uint64_t)kRiceChunk) { ok = false; break; }
            continue;
          }
          q += (uint64_t)t;
          pos += (uint64_t)t + 1;
          break;
        }
        if (!ok || pos + (uint64_t)kr > nbits) { ok = false; break; }
        const uint64_t run = (q << kr) | get_bits(rw, pos, kr);
        pos += (uint64_t)kr;
        if (run > (uint64_t)(c1 - e)) { ok = false; break; }
        e += (int64_t)run;
        if (e == c1) break;
        if (pos + (uint64_t)wv > nbits) { ok = false; break; }
        const int32_t kv = unzigzag(get_bits(rw, pos, wv) + 1u);
        pos += (uint64_t)wv;
        // the read-backs of the outputs go eight at a time (distinct elements)
        pg[npend] = elem_off(P, g, e);
        pk[npend] = kv;
        if (++npend == 8) flush();
        ++e;
      }
      flush();
      if (!ok) atomicOr(&st->corrupt, 1u);
    }
  } else if (!dense && wk > 0) {
    // entry-list corrections read the rows' outputs back: eight entries a
    // thread at a time, all eight loads issued before the first store, so that
    // the read-backs overlap (entries name distinct elements)
    constexpr int kB = 8;
    for (int64_t i0 = tid; i0 < ncorr; i0 += (int64_t)kB * NT) {
      int64_t gi[kB];
      int32_t kv[kB];
      T val[kB];
#pragma unroll
      for (int b = 0; b < kB; ++b) {
        const int64_t i = i0 + (int64_t)b * NT;
        gi[b] = -1;
        kv[b] = 0;
        if (i < ncorr) {
          const uint64_t pos = (uint64_t)i * (uint64_t)(ib + wk);
          const int64_t e = get_bits(cw, pos, ib);
          kv[b] = unzigzag(get_bits(cw, pos + ib, wk));
          if (e >= N) atomicOr(&st->corrupt, 1u);
          else gi[b] = elem_off(P, g, e);
        }
      }
#pragma unroll
      for (int b = 0; b < kB; ++b) val[b] = gi[b] >= 0 ? out[gi[b]] : T(0);
#pragma unroll
      for (int b = 0; b < kB; ++b)
        if (gi[b] >= 0) out[gi[b]] = tf<T>((T)kv[b], step_t, val[b]);
    }
  }
  __syncthreads();
  if (nesc > 0) {
    const uint32_t* ei = reinterpret_cast<const uint32_t*>(rec + lay.off_ei);
    const T* ev = reinterpret_cast<const T*>(rec + lay.off_ev);
    for (int64_t i = tid; i < nesc; i += NT) {
      const int64_t e = ei[i];
      if (e >= N) { atomicOr(&st->corrupt, 1u); continue; }
      out[elem_off(P, g, e)] = ev[i];
    }
  }
}

template <typename T, int NM>
__global__ void __launch_bounds__(kDecThreads, 3) k_decode(Plan P, const uint8_t* __restrict__ comp,
                                                           unsigned long long comp_bytes, T* __restrict__ out,
                                                           Status* st) {
  extern __shared__ __align__(16) uint32_t stage_sm[];   // kDecStageWords
  decode_block<T, NM, kDecThreads, NM == 16 && sizeof(T) == 4>(P, comp, comp_bytes, out, st, blockIdx.x, stage_sm, kDecStageWords);
}

// ---------------------------------------------------------------- float32, Gram order <= 16
// Persistent decoder of float32 plans with Gram order <= 16 and blocks of at
// most 65 536 points whose whole blocks are time-side: CTAs take blocks from a
// counter and bring each record in whole by one bulk copy, the next once the
// block is done.  Time-side blocks of rank <= 8 take the path below when their
// corrections are dense (up to 8 bits), listed (up to 4 bits, |k| <= 8) or Rice
// coded (values up to 3 bits, |k| <= 4), any other block decode_block.
//  - Listed and Rice-coded corrections go to a nibble a point in shared memory
//    first (entries by all threads, a Rice chunk a thread), so that the rows
//    add them as they write each output: no output is read back.
//  - A thread takes four neighbouring rows where lines are whole multiples of
//    16 bytes: 16-byte stores, four corrections a load, the basis read once for
//    four outputs (about 10 instructions an output; a row a thread with
//    read-backs took 34, which bound it).
//  - Three CTAs an SM (32 KB of nibbles, 41 KB of record, 80 registers) cover
//    each other's copies, scatter and Rice chains.  A byte a point with two
//    staged records (one CTA of 512 threads, or two with records up to 23 KB)
//    left the SM waiting at barriers: 1.07 and 1.71 to 2.96 ms on the two below.
// Measured: 4 GiB at 1e-3 x range (23 KB records) 1.50 -> 1.05 ms; five ragged
// variables with Rice-coded corrections (193 M points) 2.61 -> 0.99 ms.
// (out of line: the registers of the common path stay its own)
__device__ __noinline__ void decode_block_f32(const Plan& P, const uint8_t* comp, unsigned long long comp_bytes,
                                              float* out, Status* st, int64_t bi, uint32_t* stage_sm, int words) {
  decode_block<float, 16, kDecThreads>(P, comp, comp_bytes, out, st, bi, stage_sm, words);
}
constexpr int kPlaneBytes = 32768;
constexpr int kRecPad = 64;                 // readable bytes past a staged record
constexpr int kRecCap = 41920;              // bytes of a record staged beside the plane
constexpr int kRecCapAll = kPlaneBytes + kRecCap;   // ... over it (records that need no plane)
constexpr uint32_t kNoCorr = 0x88888888u;   // eight nibbles k + 8 = 8
struct DecRec {                             // one staged record, parsed by warp 0
  int r, wk, wv, kr, n, M, ncorr, nesc, mode, dense, rice, bad;
  uint32_t off_v, off_c, rice_words;
  uint32_t qbase[8];                        // word offset of column c in the record
  int wq[8];
  int64_t off_ei, off_ev;
};
enum : int { kDecSkip = 0, kDecFast = 1, kDecRaw = 2, kDecGeneric = 3 };

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// Waits at most about a second of SM clock.
__device__ __forceinline__ bool bar_wait(unsigned long long* b, unsigned parity) {
  const long long t0 = clock64();
  for (;;) {
    for (int i = 0; i < 256; ++i) {
      uint32_t ok;
      asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                   : "=r"(ok) : "r"(smem_addr(b)), "r"(parity) : "memory");
      if (ok) return true;
    }
    if (clock64() - t0 > (1ll << 31)) return false;
  }
}

// Field `i` of width w (<= 32; mask (1 << w) - 1) of a column of words; reads
// one word past the field's own.
__device__ __forceinline__ uint32_t field(const uint32_t* w, uint32_t i, int width, uint32_t mask) {
  const uint32_t pos = i * (uint32_t)width;
  const uint32_t* p = w + (pos >> 5);
  return __funnelshift_r(p[0], p[1], pos & 31u) & mask;
}

// The rows of a block: R modes, V neighbouring rows a thread, corrections from
// nowhere (CM = 0), the nibble plane (1) or the dense section (2).
template <int R, int V, int CM, int NT>
__device__ __forceinline__ void dec_rows(const Plan& P, const Geom& g, const DecRec& D, const uint32_t* rec,
                                         const float* vst, const uint8_t* plane, float delta, float step,
                                         float* __restrict__ out) {
  const int M = D.M, n = D.n, wk = D.wk;
  const int64_t tstep = P.P;
  uint32_t kmask = 0;
  const uint32_t* cw = rec;
  if (CM == 2) {
    kmask = (1u << wk) - 1u;
    cw = rec + D.off_c / 4;
  }
  for (int l = threadIdx.x * V; l < M; l += NT * V) {
    float ch[R > 0 ? R : 1][V];
#pragma unroll
    for (int c = 0; c < R; ++c) {
      const int w = D.wq[c];
      const uint32_t mask = w >= 32 ? 0xFFFFFFFFu : (1u << w) - 1u;
      const uint32_t* col = rec + D.qbase[c];
#pragma unroll
      for (int v = 0; v < V; ++v) ch[c][v] = dq<float>(unzigzag(field(col, (uint32_t)(l + v), w, mask)), delta);
    }
    float* o = out + spatial_off(P, g, l) + g.t0 * P.P;
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
      float acc[V];
#pragma unroll
      for (int v = 0; v < V; ++v) acc[v] = 0.0f;
      if (R > 0) {
        float b[R > 4 ? 8 : 4];
        *reinterpret_cast<float4*>(b) = *reinterpret_cast<const float4*>(vst + j * 8);
        if (R > 4) *reinterpret_cast<float4*>(b + 4) = *reinterpret_cast<const float4*>(vst + j * 8 + 4);
#pragma unroll
        for (int c = 0; c < R; ++c)
#pragma unroll
          for (int v = 0; v < V; ++v) acc[v] = __fmaf_rn(ch[c][v], b[c], acc[v]);
      }
      // fma(-k, -step, acc): a correction of zero adds a zero of negative sign,
      // which leaves every acc as it is, zeros of either sign among them
      if (CM == 1) {
        // (float)-k as (2^23 + 8) - (2^23 + k + 8): exact, and off the conversion pipe
        const int e = j * M + l;
        const uint32_t k4 = V == 4 ? (uint32_t)reinterpret_cast<const uint16_t*>(plane)[e >> 2]
                                   : (uint32_t)plane[e >> 1] >> ((e & 1) * 4);
#pragma unroll
        for (int v = 0; v < V; ++v)
          acc[v] = __fmaf_rn(__fsub_rn(8388616.0f, __uint_as_float(((k4 >> (4 * v)) & 15u) | 0x4B000000u)), -step, acc[v]);
      }
      if (CM == 2) {
        // V wk <= 32 bits from one unaligned word; (float)-k as above, |k| <= 128
        const uint32_t pos = (uint32_t)(j * M + l) * (uint32_t)wk;
        const uint32_t* p = cw + (pos >> 5);
        const uint32_t f = __funnelshift_r(p[0], p[1], pos & 31u);
#pragma unroll
        for (int v = 0; v < V; ++v)
          acc[v] = __fmaf_rn(__fsub_rn(8388864.0f, __int_as_float(0x4B000100 + unzigzag((f >> (v * wk)) & kmask))), -step, acc[v]);
      }
      if (V == 4) *reinterpret_cast<float4*>(o) = make_float4(acc[0], acc[V > 1 ? 1 : 0], acc[V > 2 ? 2 : 0], acc[V > 3 ? 3 : 0]);
      else *o = acc[0];
      o += tstep;
    }
  }
}
template <int V, int CM, int NT>
__device__ __forceinline__ void dec_rows_rank(const Plan& P, const Geom& g, const DecRec& D, const uint32_t* rec,
                                              const float* vst, const uint8_t* plane, float delta, float step,
                                              float* __restrict__ out) {
  switch (D.r) {
    case 0: dec_rows<0, V, CM, NT>(P, g, D, rec, vst, plane, delta, step, out); break;
    case 1: dec_rows<1, V, CM, NT>(P, g, D, rec, vst, plane, delta, step, out); break;
    case 2: dec_rows<2, V, CM, NT>(P, g, D, rec, vst, plane, delta, step, out); break;
    case 3: dec_rows<3, V, CM, NT>(P, g, D, rec, vst, plane, delta, step, out); break;
    case 4: dec_rows<4, V, CM, NT>(P, g, D, rec, vst, plane, delta, step, out); break;
    case 5: dec_rows<5, V, CM, NT>(P, g, D, rec, vst, plane, delta, step, out); break;
    case 6: dec_rows<6, V, CM, NT>(P, g, D, rec, vst, plane, delta, step, out); break;
    case 7: dec_rows<7, V, CM, NT>(P, g, D, rec, vst, plane, delta, step, out); break;
    default: dec_rows<8, V, CM, NT>(P, g, D, rec, vst, plane, delta, step, out); break;
  }
}

// Correction k (|k| <= 8, below 8) of element e into the nibble plane (once an element).
__device__ __forceinline__ void plane_put(uint32_t* plane, uint32_t e, int32_t k) {
  atomicXor(&plane[e >> 3], (((uint32_t)(k + 8) ^ 8u) & 15u) << ((e & 7u) * 4));
}

// One Rice chunk [e, c1) into the plane by one thread; false when the coded
// words do not hold it.  A code is read from one 64-bit window at its first bit
// (31 ones, a zero, kr <= 20 and wv <= 3 bits at most), so that the chain from
// one code to the next is a load, a count and a few shifts; longer runs of ones
// take the loop.
__device__ bool dec_rice_chunk(const uint32_t* __restrict__ rw, uint32_t words, uint32_t pos, int kr, int wv, int e,
                               int c1, uint32_t* plane) {
  const uint32_t nbits = words * 32u, kmask = (1u << kr) - 1u, vmask = (1u << wv) - 1u;
  if (pos >= nbits) return false;
  for (;;) {
    const uint32_t* p = rw + (pos >> 5);
    const uint32_t w0 = p[0], w1 = p[1], w2 = p[2], sh = pos & 31u;
    const uint64_t win = (uint64_t)__funnelshift_r(w0, w1, sh) | ((uint64_t)__funnelshift_r(w1, w2, sh) << 32);
    const uint32_t ones = ~(uint32_t)win;
    uint32_t q, rest;
    if (ones != 0u) {
      q = (uint32_t)__ffs(ones) - 1u;
      rest = (uint32_t)(win >> (q + 1u));
    } else {
      // 32 ones or more
      q = 32;
      for (;;) {
        const uint32_t at = pos + q;
        if (at >= nbits || q > (uint32_t)kRiceChunk) return false;
        const uint32_t* r = rw + (at >> 5);
        const uint32_t z = ~__funnelshift_r(r[0], r[1], at & 31u);
        if (z != 0u) { q += (uint32_t)__ffs(z) - 1u; break; }
        q += 32;
      }
      const uint32_t at = pos + q + 1u;
      if (at >= nbits + 32u) return false;
      const uint32_t* r = rw + (at >> 5);
      rest = __funnelshift_r(r[0], r[1], at & 31u);
    }
    const uint32_t run = (q << kr) | (rest & kmask);
    pos += q + 1u + (uint32_t)kr;
    if (pos > nbits || run > (uint32_t)(c1 - e)) return false;
    e += (int)run;
    if (e == c1) return true;
    pos += (uint32_t)wv;
    if (pos > nbits) return false;
    plane_put(plane, (uint32_t)e, unzigzag(((rest >> kr) & vmask) + 1u));
    ++e;
  }
}

// Parses and checks a staged record (warp 0).
__device__ void dec_parse(const Plan& P, const Geom& g, const uint8_t* rec, int nbytes, DecRec& D) {
  const int lane = threadIdx.x & 31;
  const uint32_t* rec32 = reinterpret_cast<const uint32_t*>(rec);
  const int r = rec[0], flags = rec[1], wk = rec[2], ib = rec[3], n = g.n;
  const uint32_t ncorr = rec32[1], nesc = rec32[2];
  const int N = (int)g.N, L = (int)g.L;
  int mode = kDecFast;
  if ((int)rec32[3] != nbytes || (flags & ~(int)(kFlagRaw | kFlagSpatial | kFlagDense | kFlagRice)) != 0) mode = kDecGeneric;
  else if (flags & kFlagRaw) mode = kDecRaw;
  else if (g.side != 0 || (flags & kFlagSpatial) || r > 8 || wk > 8 || 24 > nbytes || r > (P.rank_cap < n ? P.rank_cap : n) ||
           ib != bit_width((uint32_t)(N - 1)) || ncorr > (uint32_t)N || nesc > (uint32_t)N)
    mode = kDecGeneric;                     // refused there where it is damaged
  if (mode == kDecRaw && 16 + N * 4 > nbytes) mode = kDecGeneric;
  int w = 0, words = 0;
  if (mode == kDecFast && lane < r) {
    w = rec[16 + lane];
    words = (int)(((int64_t)L * w + 31) >> 5);
  }
  if (__any_sync(0xffffffffu, w > 32)) mode = kDecGeneric;
  int incl = words;
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const int qwords = __shfl_sync(0xffffffffu, incl, 7);
  const uint32_t off_v = 16u + (r > 0 ? 8u : 0u), off_q = off_v + (((uint32_t)(n * r) * 4u + 7u) & ~7u);
  if (lane < 8) {
    D.wq[lane] = w;
    D.qbase[lane] = off_q / 4 + (uint32_t)(incl - words);
  }
  if (lane != 0) return;
  D.mode = mode;
  if (mode != kDecFast) return;
  const int64_t dense_w = ((int64_t)N * wk + 31) >> 5, sparse_w = ((int64_t)ncorr * (ib + wk) + 31) >> 5;
  const bool dense = wk > 0 && dense_w < sparse_w, rice = (flags & kFlagRice) != 0;
  int64_t cwords = wk == 0 ? 0 : (dense ? dense_w : sparse_w);
  const int64_t off_c = (int64_t)off_q + (((int64_t)qwords * 4 + 7) & ~7ll);
  D.rice_words = 0;
  D.kr = D.wv = 0;
  if (rice) {
    if (wk == 0 || (flags & kFlagDense) || off_c + 8 > nbytes) { D.mode = kDecGeneric; return; }
    const uint32_t* cw = reinterpret_cast<const uint32_t*>(rec + off_c);
    D.rice_words = cw[0];
    D.kr = (int)(cw[1] & 0xFFu);
    D.wv = (int)((cw[1] >> 8) & 0xFFu);
    if ((cw[1] >> 16) != 0u || D.kr > kRiceMaxKr || D.wv > 3 || cw[0] > (uint32_t)nbytes) { D.mode = kDecGeneric; return; }
    cwords = 2 + (N + kRiceChunk - 1) / kRiceChunk + (int64_t)cw[0];
  } else if (dense != ((flags & kFlagDense) != 0)) {
    D.mode = kDecGeneric;
    return;
  }
  if (!dense || rice) {
    // the nibbles hold -8 .. 7, and the plane must lie beside the record
    if (wk > 4 || nbytes > kRecCap) { D.mode = kDecGeneric; return; }
  }
  D.off_ei = off_c + ((cwords * 4 + 7) & ~7ll);
  D.off_ev = D.off_ei + (((int64_t)nesc * 4 + 7) & ~7ll);
  const int64_t size = (D.off_ev + (((int64_t)nesc * 4 + 7) & ~7ll) + 15) & ~15ll;
  if (size != nbytes) { D.mode = kDecGeneric; return; }
  D.r = r;
  D.wk = wk;
  D.n = n;
  D.M = (int)g.M;
  D.ncorr = (int)ncorr;
  D.nesc = (int)nesc;
  D.dense = dense ? 1 : 0;
  D.rice = rice ? 1 : 0;
  D.off_v = off_v;
  D.off_c = (uint32_t)off_c;
}

__global__ void __launch_bounds__(kDecThreads, 3) k_decode_f32(Plan P, const uint8_t* __restrict__ comp,
                                                               unsigned long long comp_bytes, float* __restrict__ out,
                                                               Status* st, int vec, long long withhold) {
  extern __shared__ __align__(128) unsigned char dsm[];       // the record, then the plane
  constexpr int NT = kDecThreads;
  uint32_t* plane = reinterpret_cast<uint32_t*>(dsm + kRecCap + kRecPad);
  const uint8_t* rec = dsm;
  __shared__ __align__(16) float vst[16 * 8];
  __shared__ DecRec D;
  __shared__ unsigned long long full;
  __shared__ int64_t blk;
  __shared__ int bytes;                      // of the staged record (0: not staged)
  __shared__ int stop;
  const int tid = threadIdx.x;
  const uint64_t* offs = reinterpret_cast<const uint64_t*>(comp + P.offsets_pos);
  // the next block (thread 0)
  auto fetch = [&]() {
    const int64_t b = (int64_t)atomicAdd(&st->pad[0], 1ull);
    blk = b;
    bytes = 0;
    if (b >= P.nb) return;
    const uint64_t o0 = offs[b], o1 = offs[b + 1];
    if (!record_in(o0, o1, comp_bytes - (uint64_t)P.payload_pos) || (o1 & 15) != 0 || o1 - o0 > (uint64_t)kRecCapAll) return;
    const uint32_t nb = (uint32_t)(o1 - o0);
    bytes = (int)nb;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(&full)), "r"(nb) : "memory");
    if (b == withhold) return;               // test hook: nothing arrives, the wait runs out
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_addr(dsm)),
                 "l"(comp + P.payload_pos + o0), "r"(nb), "r"(smem_addr(&full))
                 : "memory");
  };
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&full)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    stop = 0;
    fetch();
  }
  __syncthreads();
  unsigned phase = 0u;
  for (;;) {
    const int64_t bi = blk;
    if (bi >= P.nb) break;
    const Geom g = block_geom(P, P.b0 + bi);
    const int nbytes = bytes;
    if (nbytes > 0) {
      if (bar_wait(&full, phase)) phase ^= 1u;
      else stop = 1;
      if (tid < 32) {
        dec_parse(P, g, rec, nbytes, D);
      } else if (nbytes <= kRecCap && rec[2] != 0 && !(rec[1] & kFlagDense)) {
        // (the plane of a record whose corrections are not dense)
        for (int i = tid - 32; i < ((int)g.N + 31) / 32; i += NT - 32)
          reinterpret_cast<uint4*>(plane)[i] = make_uint4(kNoCorr, kNoCorr, kNoCorr, kNoCorr);
      }
      {
        // basis by component, modes padded to 8 (records' own order: mode by mode)
        const int r = rec[0] < 8 ? rec[0] : 8;
        const float* vin = reinterpret_cast<const float*>(rec + 24);
        for (int i = tid; i < g.n * r; i += NT) {
          const int c = i / g.n, j = i - c * g.n;
          vst[j * 8 + c] = vin[i];
        }
      }
    } else if (tid == 0) {
      D.mode = kDecGeneric;
    }
    __syncthreads();
    if (stop) break;
    const int mode = D.mode;
    if (mode == kDecFast) {
      const double* vt = reinterpret_cast<const double*>(comp + kHdr + kVarRec * g.v);
      const float delta = __double2float_rn(vt[2]), step = __double2float_rn(vt[3]);
      const uint32_t* rec32 = reinterpret_cast<const uint32_t*>(rec);
      const uint32_t* cw = rec32 + D.off_c / 4;
      const int N = (int)g.N;
      const bool use_plane = D.wk > 0 && !(D.dense && !D.rice);
      if (use_plane) {
        if (D.rice) {
          const int nch = (N + kRiceChunk - 1) / kRiceChunk;
          for (int c = tid; c < nch; c += NT) {
            const int c1 = (c + 1) * kRiceChunk < N ? (c + 1) * kRiceChunk : N;
            if (!dec_rice_chunk(cw + 2 + nch, D.rice_words, cw[2 + c], D.kr, D.wv, c * kRiceChunk, c1, plane))
              atomicOr(&st->corrupt, 1u);
          }
        } else {
          const int ib = bit_width((uint32_t)(N - 1)), wk = D.wk, W = ib + wk;      // W <= 20
          const uint32_t em = (1u << ib) - 1u, km = (1u << wk) - 1u;
          for (int i = tid; i < D.ncorr; i += NT) {
            const uint32_t f = field(cw, (uint32_t)i, W, 0xFFFFFFFFu);
            const uint32_t e = f & em;
            if (e >= (uint32_t)N) atomicOr(&st->corrupt, 1u);
            else plane_put(plane, e, unzigzag((f >> ib) & km));
          }
        }
        __syncthreads();
      }
      const bool v4 = vec && (g.sx & 3) == 0;
      const uint8_t* pl = reinterpret_cast<const uint8_t*>(plane);
      if (use_plane) {
        if (v4) dec_rows_rank<4, 1, NT>(P, g, D, rec32, vst, pl, delta, step, out);
        else dec_rows_rank<1, 1, NT>(P, g, D, rec32, vst, pl, delta, step, out);
      } else if (D.wk > 0) {
        if (v4) dec_rows_rank<4, 2, NT>(P, g, D, rec32, vst, pl, delta, step, out);
        else dec_rows_rank<1, 2, NT>(P, g, D, rec32, vst, pl, delta, step, out);
      } else {
        if (v4) dec_rows_rank<4, 0, NT>(P, g, D, rec32, vst, pl, delta, step, out);
        else dec_rows_rank<1, 0, NT>(P, g, D, rec32, vst, pl, delta, step, out);
      }
      if (D.nesc > 0) {
        __syncthreads();
        const uint32_t* ei = reinterpret_cast<const uint32_t*>(rec + D.off_ei);
        const float* ev = reinterpret_cast<const float*>(rec + D.off_ev);
        for (int i = tid; i < D.nesc; i += NT) {
          const uint32_t e = ei[i];
          if (e >= (uint32_t)N) { atomicOr(&st->corrupt, 1u); continue; }
          out[elem_off(P, g, e)] = ev[i];
        }
      }
    } else if (mode == kDecRaw) {
      const float* vals = reinterpret_cast<const float*>(rec + 16);
      for (int64_t e = tid; e < g.N; e += NT) out[elem_off(P, g, e)] = vals[e];
    } else {
      decode_block_f32(P, comp, comp_bytes, out, st, bi, reinterpret_cast<uint32_t*>(dsm), kRecCapAll / 4);
    }
    // the next record's copy writes, through the async proxy, what this block
    // left by ordinary stores (the plane, a record staged by decode_block)
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid == 0) fetch();
    __syncthreads();
  }
  // a copy did not arrive: report it, and wait for it once more before leaving
  if (stop && tid == 0) {
    atomicOr(&st->timeout, 1u);
    bar_wait(&full, phase);
  }
}


// ---------------------------------------------------------------- verification
// acc layout (doubles): per variable v (16 doubles): [0] max_abs_err key (as
// u64), [1] n_over (u64), [2] sum_sq_err, [3] sum_sq; then stream totals at
// 16*nvars: [0] n_raw, [1] sum rank, [2] n_corr, [3] n_esc, [4] basis bytes,
// [5] coeff bytes, [6] corr bytes, [7] esc bytes, [8] raw bytes, [9] header bytes.

// The stream's composition, by the CTAs of the grid's last row (they run
// beside the points' CTAs): whole numbers, summed over a warp before the
// atomics.
__device__ void verify_stream(const Plan& P, const uint8_t* __restrict__ comp, unsigned long long comp_bytes, int es,
                              double* acc) {
  double* t = acc + 16 * P.nvars;
  const uint64_t* offs = reinterpret_cast<const uint64_t*>(comp + P.offsets_pos);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t first = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31);
  for (int64_t b0 = first; b0 < P.nb; b0 += stride) {
    const int64_t bi = b0 + (threadIdx.x & 31);
    unsigned long long n[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    if (bi < P.nb) {
      const uint64_t o0 = offs[bi], o1 = offs[bi + 1];
      if (record_in(o0, o1, comp_bytes - (uint64_t)P.payload_pos)) {
        const uint8_t* rec = comp + P.payload_pos + o0;
        const uint32_t* rec32 = reinterpret_cast<const uint32_t*>(rec);
        const int r = rec[0], flags = rec[1];
        if (flags & kFlagRaw) {
          n[0] = 1;
          n[8] = rec32[3];
        } else if (r <= kMaxN && 16 + align_up(r, 8) <= (int64_t)(o1 - o0)) {
          const Geom g = block_geom(P, P.b0 + bi);
          RecLayout lay = rec_layout(r, g.n, g.L, g.N, es, rec + 16, rec[2], rec[3], rec32[1], rec32[2]);
          if ((flags & kFlagRice) && lay.off_c + 4 <= (int64_t)(o1 - o0))
            lay = rice_layout(lay, g.N, reinterpret_cast<const uint32_t*>(rec + lay.off_c)[0], rec32[2], es);
          n[1] = (unsigned long long)r;
          n[2] = rec32[1];
          n[3] = rec32[2];
          n[4] = (unsigned long long)(lay.off_q - lay.off_v);
          n[5] = (unsigned long long)(lay.off_c - lay.off_q);
          n[6] = (unsigned long long)(lay.off_ei - lay.off_c);
          n[7] = (unsigned long long)(lay.size - lay.off_ei);
          n[9] = (unsigned long long)lay.off_v;
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 10; ++k) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) n[k] += __shfl_xor_sync(0xffffffffu, n[k], o);
      if ((threadIdx.x & 31) == 0 && n[k]) atomicAdd(&t[k], (double)n[k]);
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(256) k_verify_points(Plan P, const T* __restrict__ a, const T* __restrict__ b,
                                                       const uint8_t* comp, unsigned long long comp_bytes, double* acc) {
  const int v = blockIdx.y;
  if (v == P.nvars) {
    verify_stream(P, comp, comp_bytes, (int)sizeof(T), acc);
    return;
  }
  const double eb = reinterpret_cast<const double*>(comp + kHdr + kVarRec * v)[1];
  const bool pointwise = P.eb_type != DLS_EB_NRMSE;
  // three FP64 operations a point; the comparisons are integer ones (a NaN
  // difference counts nowhere, as in a floating comparison)
  const long long inf = 0x7FF0000000000000ll, ebb = pointwise ? __double_as_longlong(eb) : inf;
  long long mxb = 0;
  double se = 0.0, sx = 0.0;
  unsigned long long over = 0;
  const int64_t base = (int64_t)v * P.K;
#pragma unroll 4
  for (int64_t i = blockIdx.x * 256ll + threadIdx.x; i < P.K; i += (int64_t)gridDim.x * 256) {
    const double x = (double)a[base + i], y = (double)b[base + i];
    const double d = fabs(x - y);
    const long long db = __double_as_longlong(d);
    if (db <= inf) {
      mxb = db > mxb ? db : mxb;
      over += db > ebb ? 1ull : 0ull;
    }
    se = fma(d, d, se);
    sx = fma(x, x, sx);
  }
  for (int o = 16; o > 0; o >>= 1) {
    const long long m2 = __shfl_xor_sync(0xffffffffu, mxb, o);
    mxb = m2 > mxb ? m2 : mxb;
    se += __shfl_xor_sync(0xffffffffu, se, o);
    sx += __shfl_xor_sync(0xffffffffu, sx, o);
    over += __shfl_xor_sync(0xffffffffu, over, o);
  }
  const double mx = __longlong_as_double(mxb);
  if ((threadIdx.x & 31) == 0) {
    unsigned long long* u = reinterpret_cast<unsigned long long*>(acc + 16 * v);
    atomicMax(&u[0], dkey(mx));
    atomicAdd(&u[1], over);
    atomicAdd(&acc[16 * v + 2], se);
    atomicAdd(&acc[16 * v + 3], sx);
  }
}

// float32 fields: the same report with the FP64 pipe kept for what needs it.
// A point's difference is s = fl32(x - y) and its rounding error e (TwoSum,
// s + e = x - y exactly).  A point is looked at one by one, in FP64, only when
// |s| reaches the thread's running maximum (rounding is monotone, so the point
// of the largest |x - y| is among them) or the bound less a relative 2^-20, or
// is not finite: one test for four points.  The sums of squares run as
// unevaluated float pairs (x^2 = p + fma(x, x, -p) exactly where neither is
// subnormal, d^2 = s^2 + 2 s e to within e^2 <= 2^-48 s^2), two points an instruction (packed FP32), per
// batch of 1024 points of a thread; each batch is added in FP64, and one whose
// squares reach 2^117 (or with a NaN or an infinity) is summed again in FP64, as
// are all of a thread's points where its sums stay below 2^-88 without being zeros.
// Loads are float4 when the field allows (4 | K, 16-byte pointers).  Bound by the issue slots (about 20
// instructions a point; scalar FP32 with a branch a point took twice that):
// two fields of 1 GiB 0.74 -> 0.49 ms, the records' pass included.
struct FF2 {
  float2 hi, lo;
};
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ void ff2_add(FF2& f, float2 a, float2 ae) {
  const float2 s = __fadd2_rn(f.hi, a);
  const float2 bb = sub2(s, f.hi);
  const float2 err = __fadd2_rn(sub2(f.hi, sub2(s, bb)), sub2(a, bb));
  f.hi = s;
  f.lo = __fadd2_rn(f.lo, __fadd2_rn(err, ae));
}
// a^2 + 2 a e into f
__device__ __forceinline__ void ff2_square(FF2& f, float2 a, float2 two_a, float2 e) {
  const float2 p = __fmul2_rn(a, a);
  const float2 np = __fmul2_rn(p, make_float2(-1.0f, -1.0f));
  ff2_add(f, p, __ffma2_rn(two_a, e, __ffma2_rn(a, a, np)));
}
__device__ __forceinline__ void ff2_square(FF2& f, float2 a) {
  const float2 p = __fmul2_rn(a, a);
  const float2 np = __fmul2_rn(p, make_float2(-1.0f, -1.0f));
  ff2_add(f, p, __ffma2_rn(a, a, np));
}
__device__ __forceinline__ float max_nan(float a, float b) {     // a NaN when either is one
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// A thread's state that rarely changes, and its (out of line) look at one point.
struct VerRare {
  double mx, eb;
  unsigned long long over;
  float mx32, eb_lo, eb_hi;
  bool pointwise;
};
__device__ __noinline__ void verify_point(VerRare& V, float x, float y) {
  const float ad = fabsf(__fsub_rn(x, y));
  const bool plain = ad < 0x1p60f, top = !plain || ad >= V.mx32;
  const bool edge = V.pointwise && (!plain || (ad >= V.eb_lo && !(ad > V.eb_hi)));
  if (V.pointwise && plain && ad > V.eb_hi) ++V.over;
  if (!(top || edge)) return;
  const double d = fabs((double)x - (double)y);
  if (top) V.mx = fmax(V.mx, d);
  if (ad > V.mx32) V.mx32 = ad;
  if (edge && d > V.eb) ++V.over;
}
// Below kPairsMost every |x| and |s| of a batch is below 2^59, every |y| below 2^60.
constexpr float kPairsMost = 0x1p117f;
// Below 2^-126 a square or its residual is off by up to 2^-150, three a point: the
// pairs' sum over a thread's batches (sixteen of them for 5 G points) is exact to
// 2^-46 of it from kPairsLeast on.
constexpr double kPairsLeast = 0x1p-88;
__device__ __noinline__ void verify_sums_fp64(const float* __restrict__ a, const float* __restrict__ b, int64_t i, int64_t n,
                                              int64_t stride, int width, double* se, double* sx) {
  for (int64_t k = 0; k < n; ++k, i += stride)
    for (int c = 0; c < width; ++c) {
      const double x = (double)a[i * width + c], y = (double)b[i * width + c], d = fabs(x - y);
      *se = fma(d, d, *se);
      *sx = fma(x, x, *sx);
    }
}
// A thread's sums again in FP64 where one is below kPairsLeast, unless that is a
// sum of zeros (`seen`: differences have been seen; the values are read again).
// (Once a thread: the same test a batch took 1 to 2% of the kernel.)
__device__ __noinline__ void verify_sums_small(const float* __restrict__ a, const float* __restrict__ b, int64_t i, int64_t n,
                                               int64_t stride, int width, bool seen, double* se, double* sx) {
  if (!(*se < kPairsLeast && seen)) {
    uint32_t any = 0u;
#pragma unroll 8
    for (int64_t k = 0; k < n; ++k)
      for (int c = 0; c < width; ++c) any |= __float_as_uint(a[(i + k * stride) * width + c]) << 1;
    if (any == 0u) return;
  }
  *se = *sx = 0.0;
  verify_sums_fp64(a, b, i, n, stride, width, se, sx);
}

// Four CTAs an SM: at 70 registers, three of them, 1 GiB took 644 us a call
// instead of 537.
__global__ void __launch_bounds__(256, 4) k_verify_points_f32(Plan P, const float* __restrict__ a,
                                                           const float* __restrict__ b, const uint8_t* comp,
                                                           unsigned long long comp_bytes, double* acc, int vec4) {
  const int v = blockIdx.y;
  if (v == P.nvars) {
    verify_stream(P, comp, comp_bytes, 4, acc);
    return;
  }
  VerRare V;
  V.eb = reinterpret_cast<const double*>(comp + kHdr + kVarRec * v)[1];
  V.pointwise = P.eb_type != DLS_EB_NRMSE;
  V.mx = 0.0;
  V.over = 0;
  V.mx32 = 0.0f;
  // |s| below this needs no look: below the bound with room for the roundings, and below the maximum so far
  const float eb_lo = V.pointwise ? __double2float_rd(V.eb * (1.0 - 0x1p-20)) : INFINITY;
  V.eb_lo = eb_lo;
  V.eb_hi = __double2float_ru(V.eb * (1.0 + 0x1p-20));
  float thr = 0.0f;
  double se = 0.0, sx = 0.0;
  const float2 zero = make_float2(0.0f, 0.0f);
  FF2 fe{zero, zero}, fx{zero, zero};
  auto pair = [&](float2 x, float2 y) -> float2 {
    const float2 s = sub2(x, y);
    const float2 bb = sub2(s, x);
    const float2 e = sub2(sub2(x, sub2(s, bb)), __fadd2_rn(y, bb));
    ff2_square(fe, s, __fadd2_rn(s, s), e);
    ff2_square(fx, x);
    return s;
  };
  auto flush = [&](const float* a0, const float* b0, int64_t i, int64_t n, int64_t stride, int width) {
    const float h = (fe.hi.x + fe.hi.y) + (fx.hi.x + fx.hi.y) + (fe.lo.x + fe.lo.y) + (fx.lo.x + fx.lo.y);
    if (fabsf(h) < kPairsMost) {
      se += ((double)fe.hi.x + (double)fe.lo.x) + ((double)fe.hi.y + (double)fe.lo.y);
      sx += ((double)fx.hi.x + (double)fx.lo.x) + ((double)fx.hi.y + (double)fx.lo.y);
    } else {
      verify_sums_fp64(a0, b0, i, n, stride, width, &se, &sx);
    }
    fe = FF2{zero, zero};
    fx = FF2{zero, zero};
  };
  const int64_t base = (int64_t)v * P.K;
  const int64_t stride = (int64_t)gridDim.x * 256;
  if (vec4) {
    // four points a load; batches of 256 loads (1024 points)
    const float4* a4 = reinterpret_cast<const float4*>(a + base);
    const float4* b4 = reinterpret_cast<const float4*>(b + base);
    const int64_t K4 = P.K / 4;
    int64_t i = blockIdx.x * 256ll + threadIdx.x;
    auto four = [&](const float4& x, const float4& y) {
      const float2 s0 = pair(make_float2(x.x, x.y), make_float2(y.x, y.y));
      const float2 s1 = pair(make_float2(x.z, x.w), make_float2(y.z, y.w));
      const float m = max_nan(max_nan(fabsf(s0.x), fabsf(s0.y)), max_nan(fabsf(s1.x), fabsf(s1.y)));
      if (!(m < thr) && m != 0.0f) {
        verify_point(V, x.x, y.x);
        verify_point(V, x.y, y.y);
        verify_point(V, x.z, y.z);
        verify_point(V, x.w, y.w);
        thr = fminf(V.mx32, eb_lo);
      }
    };
    while (i < K4) {
      const int64_t i0 = i;
      int n = 0;
      for (; n < 256 && i + 3 * stride < K4; n += 4, i += 4 * stride) {
        float4 x[4], y[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) { x[k] = __ldcs(a4 + i + k * stride); y[k] = __ldcs(b4 + i + k * stride); }
#pragma unroll
        for (int k = 0; k < 4; ++k) four(x[k], y[k]);
      }
      if (n < 256)
        for (; i < K4; ++n, i += stride) four(a4[i], b4[i]);
      flush(a + base, b + base, i0, n, stride, 4);
    }
  } else {
    int64_t i = blockIdx.x * 256ll + threadIdx.x;
    while (i < P.K) {
      const int64_t i0 = i;
      int n = 0;
      for (; n < 1024 && i < P.K; n += 2, i += 2 * stride) {
        // (a missing second point is a pair of zeros)
        const bool two = i + stride < P.K;
        const float2 x = make_float2(a[base + i], two ? a[base + i + stride] : 0.0f);
        const float2 y = make_float2(b[base + i], two ? b[base + i + stride] : 0.0f);
        const float2 s = pair(x, y);
        const float m = max_nan(fabsf(s.x), fabsf(s.y));
        if (!(m < thr) && m != 0.0f) {
          verify_point(V, x.x, y.x);
          if (two) verify_point(V, x.y, y.y);
          thr = fminf(V.mx32, eb_lo);
        }
      }
      const int64_t left = (P.K - i0 + stride - 1) / stride;
      flush(a + base, b + base, i0, n < left ? n : left, stride, 1);
    }
  }
  if ((se < kPairsLeast && V.mx32 > 0.0f) || sx < kPairsLeast) {
    const int64_t i0 = blockIdx.x * 256ll + threadIdx.x, end = vec4 ? P.K / 4 : P.K;
    if (i0 < end)
      verify_sums_small(a + base, b + base, i0, (end - i0 + stride - 1) / stride, stride, vec4 ? 4 : 1, V.mx32 > 0.0f, &se, &sx);
  }
  double mx = V.mx;
  unsigned long long over = V.over;
  for (int o = 16; o > 0; o >>= 1) {
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    se += __shfl_xor_sync(0xffffffffu, se, o);
    sx += __shfl_xor_sync(0xffffffffu, sx, o);
    over += __shfl_xor_sync(0xffffffffu, over, o);
  }
  if ((threadIdx.x & 31) == 0) {
    unsigned long long* u = reinterpret_cast<unsigned long long*>(acc + 16 * v);
    atomicMax(&u[0], dkey(mx));
    atomicAdd(&u[1], over);
    atomicAdd(&acc[16 * v + 2], se);
    atomicAdd(&acc[16 * v + 3], sx);
  }
}

}  // namespace

int launch_decode(const Plan& p, const void* d_comp, unsigned long long comp_bytes, void* d_out,
                        Status* st, cudaStream_t s) {
  if (p.nb == 0) return DLS_OK;
  const uint8_t* c = (const uint8_t*)d_comp;
  const int64_t mblk = (int64_t)p.block[0] * p.block[1] * p.block[2], nblk = mblk * p.block[3];
  // (plans whose whole blocks are space-side have no use for the staged records:
  // 67 M points in blocks of 4 x 2 x 1 x 16: 9514 us through it, 6094 without)
  if (p.dtype == DLS_F32 && p.nmax <= 16 && nblk <= 2 * kPlaneBytes && mblk >= p.block[3]) {
    int dev = 0, sms = 152;
    const int smem = kRecCapAll + kRecPad;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(k_decode_f32, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
      return DLS_ERR_CUDA;
    // 16-byte stores need whole x lines and planes of 16-byte multiples
    const int vec = p.dims[0] % 4 == 0 && p.block[0] % 4 == 0 && ((uintptr_t)d_out & 15) == 0 ? 1 : 0;
    const int64_t most = (int64_t)sms * 3;
    k_decode_f32<<<(unsigned)(p.nb < most ? p.nb : most), kDecThreads, smem, s>>>(p, c, comp_bytes, (float*)d_out, st, vec,
                                                                                   fault_withheld_record());
    return cudaGetLastError() == cudaSuccess ? DLS_OK : DLS_ERR_CUDA;
  }
  const unsigned grid = (unsigned)p.nb;
  const int sm = kDecStageWords * 4;
  // the stage buffer is above the 48 KB default: opt in before each launch
  auto go = [&](auto kern, auto* outp) -> bool {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, sm) != cudaSuccess) return false;
    kern<<<grid, kDecThreads, sm, s>>>(p, c, comp_bytes, outp, st);
    return true;
  };
  bool ok;
  if (p.dtype == DLS_F32)
    ok = p.nmax <= 16 ? go(k_decode<float, 16>, (float*)d_out) : go(k_decode<float, 32>, (float*)d_out);
  else
    ok = p.nmax <= 16 ? go(k_decode<double, 16>, (double*)d_out) : go(k_decode<double, 32>, (double*)d_out);
  return ok && cudaGetLastError() == cudaSuccess ? DLS_OK : DLS_ERR_CUDA;
}

int launch_verify(const Plan& p, const void* d_orig, const void* d_recon, const void* d_comp,
                  unsigned long long comp_bytes, double* acc, cudaStream_t s) {
  // the points' CTAs, all resident at once (each a few batches), and a row for the stream's records
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return DLS_ERR_CUDA;
  const int64_t want = cdiv(p.K, 4096), most = (int64_t)sms * 8;
  const dim3 grid((unsigned)(want < 1 ? 1 : want < most ? want : most), (unsigned)p.nvars + 1);
  if (p.dtype == DLS_F32)
    k_verify_points_f32<<<grid, 256, 0, s>>>(p, (const float*)d_orig, (const float*)d_recon, (const uint8_t*)d_comp,
                                             comp_bytes, acc,
                                             (p.K % 4 == 0 && ((uintptr_t)d_orig & 15) == 0 &&
                                              ((uintptr_t)d_recon & 15) == 0) ? 1 : 0);
  else
    k_verify_points<double><<<grid, 256, 0, s>>>(p, (const double*)d_orig, (const double*)d_recon, (const uint8_t*)d_comp,
                                                 comp_bytes, acc);
  return cudaGetLastError() == cudaSuccess ? DLS_OK : DLS_ERR_CUDA;
}

}  // namespace dls
