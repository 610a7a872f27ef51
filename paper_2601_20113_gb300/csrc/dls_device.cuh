// Device helpers shared by the kernels (exact conversions, bit packing, block scans).
#pragma once

#include "dls_internal.cuh"

namespace dls {

// The FP64 pipe issues about two lanes a clock and SM (an FP64 instruction,
// a conversion from float included, holds a quarter of the SM for 64 clocks),
// so what integers can do is done with them.
// (double)x exactly where x is finite; infinities and NaNs come out finite:
// callers screen them.
__device__ __forceinline__ double widen(float x) {
  const uint32_t u = __float_as_uint(x);
  if ((u & 0x7F800000u) == 0u) return (double)x;       // zeros and subnormals
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(u << 29));
}
// (double)x exactly whatever x is, for values that nothing has screened (a
// decoded value may have overflowed): widen with the exponent of infinities and
// NaNs kept at its largest.
__device__ __forceinline__ double widen_any(float x) {
  const uint32_t u = __float_as_uint(x);
  if ((u & 0x7F800000u) != 0x7F800000u) return widen(x);
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + 0x70000000u)), (int)(u << 29));
}
__device__ __forceinline__ double widen_any(double x) { return x; }
// widen for passes that stream their input: a subnormal is scaled by 2^32
// first (exactly) instead of converted, since the compiler runs the conversion
// for every value and selects (the statistics pass on 43 M floats: 196 us with
// it, 96 without; the norm pass on 34 M: 152 and 73).  In chains of dependent FMAs
// the extra integer work costs more (the patch kernel: 1576 us with widen,
// 1757 with this one).
__device__ __forceinline__ double widen_stream(float x) {
  const bool small = (__float_as_uint(x) & 0x7F800000u) == 0u;
  const uint32_t u = __float_as_uint(small ? __fmul_rn(x, 4294967296.0f) : x), m = u & 0x7FFFFFFFu;
  const uint32_t bias = small ? 0x38000000u - (32u << 20) : 0x38000000u;
  const uint32_t hi = m ? (m >> 3) + bias : 0u;
  return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(u << 29));
}
__device__ __forceinline__ double widen_stream(double x) { return x; }
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ bool not_finite(float x) { return (__float_as_uint(x) & 0x7F800000u) == 0x7F800000u; }
__device__ __forceinline__ bool not_finite(double x) { return (__double2hiint(x) & 0x7FF00000) == 0x7FF00000; }
// |x| < b for a finite b >= 0, on the bit patterns (false for a NaN x).
__device__ __forceinline__ bool mag_below(double x, double b) {
  return (__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFll) < __double_as_longlong(b);
}
// |x| > b for b >= 0, likewise (true for a NaN x).
__device__ __forceinline__ bool mag_above(double x, double b) {
  return (__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFll) > __double_as_longlong(b);
}

// Word w of a bit stream whose element l (value val(l), width wdt) sits at bit l*wdt.
template <typename F>
__device__ __forceinline__ uint32_t compose_word(int64_t w, int wdt, int64_t count, F val) {
  const int64_t b0 = w * 32;
  int64_t l = b0 / wdt;
  uint32_t word = 0;
  for (; l < count; ++l) {
    const int64_t pos = l * wdt;
    if (pos >= b0 + 32) break;
    const uint32_t z = val(l);
    const int64_t sh = pos - b0;
    if (sh >= 0) word |= (uint32_t)((uint64_t)z << sh);
    else word |= (uint32_t)(z >> (-sh));
  }
  return word;
}

__device__ __forceinline__ void or_bits(uint32_t* words, uint64_t pos, uint32_t val, int width) {
  if (width == 0) return;
  const uint64_t wi = pos >> 5;
  const int sh = (int)(pos & 31);
  const uint64_t v = (uint64_t)val << sh;
  atomicOr(&words[wi], (uint32_t)v);
  if (sh + width > 32) atomicOr(&words[wi + 1], (uint32_t)(v >> 32));
}

// Block-wide exclusive scan of one int per thread (all threads must call);
// returns the exclusive prefix and writes the tile total to *total.
__device__ __forceinline__ int block_excl_scan(int v, int* sh_warp, int* total) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sh_warp[warp] = x;
  __syncthreads();
  if (warp == 0) {
    int s = lane < (int)(blockDim.x / 32) ? sh_warp[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    sh_warp[lane] = s;
  }
  __syncthreads();
  const int excl = (warp > 0 ? sh_warp[warp - 1] : 0) + x - v;
  *total = sh_warp[blockDim.x / 32 - 1];
  __syncthreads();
  return excl;
}

}  // namespace dls
