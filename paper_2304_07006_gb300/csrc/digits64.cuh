// Digits of FP64 values for the tensor-core FP64 contraction (gemm64_tc.cu): a row whose largest
// magnitude is below 2^e is written as x = 2^e sum_d x_d 2^(-8 - 9 d), d = 0..7, |x_d| <= 2^8, each
// digit exact in fp16: 71 bits below the row's maximum.  A value may carry a further power of 2, 2^s (the
// common scale of its index k, taken out of the other operand).  Integer arithmetic on the bit patterns only.
#pragma once
#include <cuda_fp16.h>
#include <stdint.h>

#include "xtc_internal.cuh"

namespace xtc {

// Largest of the 32-bit values of a CTA of n warps (n <= 32), to every thread.
__device__ __forceinline__ int block_max(int v, int* scratch) {
  v = __reduce_max_sync(0xffffffffu, v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = v;
  __syncthreads();
  const int n = blockDim.x >> 5;
  for (int w = 0; w < n; ++w) v = max(v, scratch[w]);
  return v;
}

// Biased exponent of a subnormal value.  Out of line: inlined it is predicated and issues for every value (464 us and not
// 435 for the left operand of K at 30 orbitals and 8,000 points).
static __device__ __noinline__ int d64_subnormal_exponent(int hi, int lo) { return hi ? 12 - __clz(hi) : -20 - __clz(lo); }

// Biased exponent of x 2^s, to be maximised over a row: 0 for x = 0, D64_NONFINITE for infinities and NaN.  That of a
// subnormal value is its own, down to -51: a density of 1e-320 at a far point, brought up by its point's scale, would
// otherwise count for up to 2^52 times its size, and its row lose as many bits.
constexpr int D64_BIAS = 1 << 16;
__device__ __forceinline__ int d64_key(double x, int s) {
  const int hi = __double2hiint(x) & 0x7fffffff, lo = __double2loint(x);
  if ((hi | lo) == 0 || s == D64_NO_SCALE) return 0;
  const int ex = hi >> 20;
  if (ex == 0) return d64_subnormal_exponent(hi, lo) + s + D64_BIAS;
  return ex == 0x7ff ? D64_NONFINITE : ex + s + D64_BIAS;
}
// Exponent e of a row (every |x 2^s| < 2^e) from the largest key.
__device__ __forceinline__ int d64_exponent(int key) {
  return key >= D64_NONFINITE ? D64_NONFINITE : (key == 0 ? 0 : key - D64_BIAS - 1022);
}

// x 2^(s + 71 - e) as an integer (rounded to nearest, ties away), plus 256 in every digit but the first:
// digit d >= 1 is then the 9-bit field at bit 9 (7 - d) minus 256, digit 0 what is left at bit 63.
struct Fixed72 {
  unsigned long long low;   // 63 bits: digits 1..7
  int top;                  // digit 0
};
__device__ __forceinline__ Fixed72 d64_fixed(double x, int s, int e) {
  constexpr unsigned long long bias = 256ull * (((1ull << 63) - 1) / 511ull);
  static_assert(((1ull << 63) - 1) % 511 == 0, "256 in seven digits");
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
  const int ex = static_cast<int>(b >> 52) & 0x7ff;
  const unsigned long long m = (b & 0xfffffffffffffull) | (ex ? 1ull << 52 : 0ull);
  const int sh = max(ex, 1) - 1004 - e + s;   // at most 18, subnormal values at most 70 (the value is below 2^71)
  unsigned long long lo = 0, hi = 0;
  if (sh >= 64) {
    hi = m << (sh - 64);
  } else if (sh > 0) {
    lo = m << sh;
    hi = m >> (64 - sh);
  } else if (sh > -54) {
    lo = sh ? (m + (1ull << (-sh - 1))) >> -sh : m;
  }
  if (static_cast<long long>(b) < 0) {
    hi = ~hi + (lo == 0);
    lo = 0ull - lo;
  }
  const unsigned long long t = lo + bias;
  hi += t < lo;
  return {t & ((1ull << 63) - 1), static_cast<int>(static_cast<long long>((hi << 1) | (t >> 63)))};
}

// The digits of four values with consecutive k, plane d at out + d * plane (8-byte aligned).
__device__ __forceinline__ void d64_store_digits(const double (&v)[4], const int (&s)[4], int e, uint16_t* out,
                                                 int64_t plane) {
  Fixed72 t[4];
#pragma unroll
  for (int q = 0; q < 4; ++q)
    t[q] = e >= D64_NONFINITE || s[q] == D64_NO_SCALE ? d64_fixed(0.0, 0, 0) : d64_fixed(v[q], s[q], e);
  const __half2 off = __halves2half2(__ushort_as_half(0x6500), __ushort_as_half(0x6500));  // 1280 = 1024 + 256
#pragma unroll
  for (int d = 0; d < D64_PLANES; ++d) {
    uint32_t f[4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      f[q] = d == 0 ? static_cast<uint32_t>(t[q].top + 256) : static_cast<uint32_t>(t[q].low >> (9 * (7 - d))) & 511u;
    // 0x6400 + f is the fp16 value 1024 + f
    uint32_t h[2] = {0x64006400u + f[0] + (f[1] << 16), 0x64006400u + f[2] + (f[3] << 16)};
    uint2 w;
    const __half2 a = __hsub2(*reinterpret_cast<__half2*>(&h[0]), off), b = __hsub2(*reinterpret_cast<__half2*>(&h[1]), off);
    w.x = *reinterpret_cast<const uint32_t*>(&a);
    w.y = *reinterpret_cast<const uint32_t*>(&b);
    *reinterpret_cast<uint2*>(out + d * plane) = w;
  }
}

}  // namespace xtc
