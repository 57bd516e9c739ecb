// Preparation kernels, the FP64 SIMT form of steps (a)+(b) (the allocation-free call), and the final kernels
// (Delta U unpacking, the one-body correction and the constant of Appendix B).
#include <algorithm>

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "jastrow_coef.cuh"
#include "simt_pack.cuh"
#include "xtc_internal.cuh"

namespace xtc {
namespace {

__device__ __forceinline__ int pair_of(int p, int q, int N) {
  // packed index of the unordered pair {p, q}
  const int a = min(p, q), b = max(p, q);
  return a * N - a * (a - 1) / 2 + (b - a);
}

// ------------------------------------------------------------------ inner-point tables
__global__ void jtab_kernel(const double* __restrict__ grid, int64_t n_grid, int64_t n_pad,
                            const JastrowParams* __restrict__ jp, int n_nuc, int js, float* __restrict__ jtab) {
  const int64_t j = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (j >= n_pad) return;
  double x = 1.0e3, y = 1.0e3, z = 1.0e3;  // padding points: far away and finite (their rho is zero)
  if (j < n_grid) {
    x = grid[3 * j];
    y = grid[3 * j + 1];
    z = grid[3 * j + 2];
  }
  // Points j = 2k and 2k+1 share a record of 2 js floats, each field stored as an adjacent (even,
  // odd) pair so that one 16-byte load yields two packed fields:
  //   x_hi y_hi | z_hi x_lo | y_lo z_lo | a_0 a_1 | a_2 a_3 | ...      (each entry = [j even, j odd])
  // with x = x_hi + x_lo (differences of nearby points keep FP64-level accuracy in FP32) and
  // a_I = |r_j - R_I| / (1 + |r_j - R_I|); js = 12 holds 4 nuclei, js = 16 holds 8 (+ 2 zero
  // fields); entries past the last nucleus are zero.
  float* o = jtab + (j >> 1) * 2 * js + (j & 1);
  const float xh = static_cast<float>(x), yh = static_cast<float>(y), zh = static_cast<float>(z);
  float f[16] = {xh, yh, zh, static_cast<float>(x - static_cast<double>(xh)),
                 static_cast<float>(y - static_cast<double>(yh)), static_cast<float>(z - static_cast<double>(zh))};
  for (int k = 6; k < 16; ++k) f[k] = 0.0f;
  for (int I = 0; I < n_nuc && I < js - 6 && I < 8; ++I) {
    const double dx = x - jp->nuc[I][0], dy = y - jp->nuc[I][1], dz = z - jp->nuc[I][2];
    const double d = sqrt(dx * dx + dy * dy + dz * dz);
    f[6 + I] = static_cast<float>(d / (1.0 + d));
  }
  for (int k = 0; k < js && k < 16; ++k) o[2 * k] = f[k];
}

__global__ void transpose_phi_kernel(const double* __restrict__ phi, int64_t n_grid, int64_t n_pad, int N,
                                     double* __restrict__ phiT) {
  __shared__ double tile[32][33];
  const int64_t j0 = blockIdx.x * 32ll;
  const int p0 = blockIdx.y * 32;
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    const int64_t j = j0 + k;
    const int p = p0 + threadIdx.x;
    tile[k][threadIdx.x] = (j < n_grid && p < N) ? phi[j * N + p] : 0.0;
  }
  __syncthreads();
  for (int k = threadIdx.y; k < 32; k += blockDim.y) {
    const int p = p0 + k;
    const int64_t j = j0 + threadIdx.x;
    if (p < N && j < n_pad) phiT[p * n_pad + j] = tile[threadIdx.x][k];
  }
}

__global__ void check_finite_kernel(const double* __restrict__ x, int64_t n, int* flag) {
  int bad = 0;
  for (int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; k < n;
       k += static_cast<int64_t>(gridDim.x) * blockDim.x)
    bad |= !isfinite(x[k]);
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 1);
}

// ------------------------------------------------------------------ pair products rho
// colmax[pq] = max_j |w_j phi_p(j) phi_q(j)| (as float bits; values are non-negative)
// power-of-2 exponent that brings the column maximum near 2^14 (fp16 split); 0 when unscaled
__device__ __forceinline__ int col_exponent(const unsigned int* colmax, int pq, bool scale) {
  if (!scale) return 0;
  const float m = __uint_as_float(colmax[pq]);
  if (!(m > 0.0f)) return 0;
  int e;
  frexpf(m, &e);           // m = f * 2^e, f in [0.5, 1)
  return min(max(14 - e, -60), 60);
}

// Orbitals and weights as FP32 pairs hi + lo (hi = the value rounded to FP32, lo = the FP32
// rounding of the rest): row r < n_orb of dst is phi_r, row n_orb the weights; dst[part][row][j].
__global__ void split_phi_f32_kernel(const double* __restrict__ phiT, const double* __restrict__ w, int64_t n_grid,
                                     int64_t n_pad, int n_orb, float* __restrict__ dst) {
  const int64_t rows = static_cast<int64_t>(n_orb) + 1, total = rows * n_pad;
  for (int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; k < total;
       k += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t r = k / n_pad, j = k % n_pad;
    const double v = r < n_orb ? phiT[k] : (j < n_grid ? w[j] : 0.0);
    const float hi = static_cast<float>(v);
    dst[k] = hi;
    dst[total + k] = static_cast<float>(v - static_cast<double>(hi));
  }
}

// w phi_p phi_q from the FP32 pairs of split_phi_f32_kernel as an unevaluated sum rh + rl (error-
// free products by fma, then one renormalisation): about 2^-44 of the value, on the FP32 pipes.
__device__ __forceinline__ void rho_pair_f32(float ah, float al, float bh, float bl, float wh, float wl, float& rh,
                                             float& rl) {
  const float xh = ah * bh;
  const float xl = fmaf(ah, bh, -xh) + fmaf(ah, bl, al * bh);
  const float yh = xh * wh;
  const float yl = fmaf(xh, wh, -yh) + fmaf(xh, wl, xl * wh);
  rh = yh + yl;
  rl = yl - (rh - yh);
}

// The pair products are taken with p fixed in a CTA and a run over q >= p: phi_p and w stay in registers
// and each product loads phi_q alone (16 bytes a point pair).  With one warp per pair and 64 points, every
// value loaded all three factors and wrote 2 bytes per lane: 20 ms for N = 200 and 200,000 points (24 GB),
// 4 bytes per lane and these loops 5 ms, against 3.7 ms at the copy rate.

// Largest |rho| of each pair over the grid (FP32; it only picks the pair's power-of-2 scale): CTA p =
// blockIdx.y, four points per thread.
constexpr int RC_POINTS = 1024;
__global__ void __launch_bounds__(256) rho_colmax_f32_kernel(const float* __restrict__ f32, int64_t n_pad, int n_orb,
                                                             unsigned int* __restrict__ colmax) {
  extern __shared__ unsigned int cmax[];  // [n_orb]
  const int p = blockIdx.y;
  const int64_t j = static_cast<int64_t>(blockIdx.x) * RC_POINTS + 4 * threadIdx.x;
  const int64_t total = (static_cast<int64_t>(n_orb) + 1) * n_pad;
  const bool in = j < n_pad;   // n_pad is a multiple of 4; padded points have zero weight
  const int64_t jj = in ? j : 0;
  auto load = [&](int64_t row, float4& hi, float4& lo) {
    hi = __ldg(reinterpret_cast<const float4*>(f32 + row * n_pad + jj));
    lo = __ldg(reinterpret_cast<const float4*>(f32 + total + row * n_pad + jj));
  };
  for (int q = p + threadIdx.x; q < n_orb; q += 256) cmax[q] = 0;
  __syncthreads();
  float4 ah, al, wh, wl;
  load(p, ah, al);
  load(n_orb, wh, wl);
#pragma unroll 2
  for (int q = p; q < n_orb; ++q) {
    float4 bh, bl;
    load(q, bh, bl);
    float rh[4], rl;
    rho_pair_f32(ah.x, al.x, bh.x, bl.x, wh.x, wl.x, rh[0], rl);
    rho_pair_f32(ah.y, al.y, bh.y, bl.y, wh.y, wl.y, rh[1], rl);
    rho_pair_f32(ah.z, al.z, bh.z, bl.z, wh.z, wl.z, rh[2], rl);
    rho_pair_f32(ah.w, al.w, bh.w, bl.w, wh.w, wl.w, rh[3], rl);
    const float m = fmaxf(fmaxf(fabsf(rh[0]), fabsf(rh[1])), fmaxf(fabsf(rh[2]), fabsf(rh[3])));
    const unsigned int bits = __reduce_max_sync(0xffffffffu, in ? __float_as_uint(m) : 0u);
    if ((threadIdx.x & 31) == 0) atomicMax(cmax + q, bits);
  }
  __syncthreads();
  const int base = p * n_orb - p * (p - 1) / 2 - p;
  for (int q = p + threadIdx.x; q < n_orb; q += 256)
    if (cmax[q]) atomicMax(colmax + base + q, cmax[q]);
}

__global__ void rho_colexp_kernel(const unsigned int* __restrict__ colmax, int n_pair, int* __restrict__ colexp) {
  const int pq = blockIdx.x * blockDim.x + threadIdx.x;
  if (pq < n_pair) colexp[pq] = col_exponent(colmax, pq, true);
}

// fp16 (2 parts, exact split): a warp takes two runs of 64 points (KD = 4: one of 128) and, with p =
// blockIdx.y fixed, the pairs (p, q), q >= p; lane t holds points 2 t and 2 t + 1 of every 64.  An accumulation
// range of the GEMM (32 KD points: half a warp's points, a warp's, or two runs) shares one quantum (largest
// |value| of the range, `bits` bits).  rho = rh + rl in FP32 pairs (rho_pair_f32); hi = rh rounded to the
// quantum (exact), lo = fp16((rh - hi) + rl), whose
// rounding error is far below fp16's.  Layout: 128-byte runs of 64 points of one part,
// [pq][j / 64][part][j % 64]; then the plane [pq][j] of the value rounded to fp16.
constexpr int RS_POINTS = 8 * 128;  // points per CTA of 8 warps
template <int KD>
__global__ void __launch_bounds__(256) rho_split_f16_kernel(const float* __restrict__ f32, int64_t n_pad, int n_orb,
                                                            int n_pair, const int* __restrict__ colexp, int bits,
                                                            uint16_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int p = blockIdx.y;
  const int64_t j0 = static_cast<int64_t>(blockIdx.x) * RS_POINTS + (threadIdx.x >> 5) * 128;
  if (j0 >= n_pad) return;  // whole warp: n_pad is a multiple of 128
  const int64_t total = (static_cast<int64_t>(n_orb) + 1) * n_pad;
  const float* base = f32 + j0 + 2 * lane;
  float2 ah[2], al[2], wh[2], wl[2];
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    ah[g] = __ldg(reinterpret_cast<const float2*>(base + p * n_pad + 64 * g));
    al[g] = __ldg(reinterpret_cast<const float2*>(base + total + p * n_pad + 64 * g));
    wh[g] = __ldg(reinterpret_cast<const float2*>(base + n_orb * n_pad + 64 * g));
    wl[g] = __ldg(reinterpret_cast<const float2*>(base + total + n_orb * n_pad + 64 * g));
  }
  uint16_t* out16 = out + static_cast<int64_t>(n_pair) * 2 * n_pad;  // the fp16(rho) plane
  const int64_t pair0 = p * n_orb - static_cast<int64_t>(p) * (p - 1) / 2 - p;
#pragma unroll 2
  for (int q = p; q < n_orb; ++q) {
    const int64_t pq = pair0 + q;
    const float sc = pow2f(__ldg(colexp + pq));  // |e| <= 60: exact scaling
    float2 vh[2], vl[2];
    unsigned int m[2];
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const float2 bh = __ldg(reinterpret_cast<const float2*>(base + q * n_pad + 64 * g));
      const float2 bl = __ldg(reinterpret_cast<const float2*>(base + total + q * n_pad + 64 * g));
      float rh, rl;
      rho_pair_f32(ah[g].x, al[g].x, bh.x, bl.x, wh[g].x, wl[g].x, rh, rl);
      vh[g].x = rh * sc;
      vl[g].x = rl * sc;
      rho_pair_f32(ah[g].y, al[g].y, bh.y, bl.y, wh[g].y, wl[g].y, rh, rl);
      vh[g].y = rh * sc;
      vl[g].y = rl * sc;
      m[g] = __float_as_uint(fmaxf(fabsf(vh[g].x), fabsf(vh[g].y)));
    }
    if (KD == 4) {
      m[0] = m[1] = __reduce_max_sync(0xffffffffu, max(m[0], m[1]));
    } else {
#pragma unroll
      for (int g = 0; g < 2; ++g) m[g] = __reduce_max_sync(KD == 2 ? 0xffffffffu : (lane < 16 ? 0xffffu : 0xffff0000u), m[g]);
    }
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const int qe = exact_quantum(__uint_as_float(m[g]), bits);
      float hx = 0.0f, hy = 0.0f;
      if (qe >= -24) {  // both products exact (powers of 2)
        const float up = pow2f(-qe), down = pow2f(qe);
        hx = rintf(vh[g].x * up) * down;
        hy = rintf(vh[g].y * up) * down;
      }
      const int64_t o = pq * 2 * n_pad + 2 * (j0 + 64 * g) + 2 * lane;
      const __half2 h = __floats2half2_rn(hx, hy);                                      // exact: at most 10 bits
      const __half2 l = __floats2half2_rn((vh[g].x - hx) + vl[g].x, (vh[g].y - hy) + vl[g].y);  // v - h is exact
      *reinterpret_cast<__half2*>(out + o) = h;
      *reinterpret_cast<__half2*>(out + o + 64) = l;
      *reinterpret_cast<__half2*>(out16 + pq * n_pad + j0 + 64 * g + 2 * lane) = __floats2half2_rn(vh[g].x, vh[g].y);
    }
  }
}

// bf16 (3 parts): per-element split with a plain power-of-2 scale of 1 (no exact ranges), one
// plane per part: [part][pq][j].
__global__ void rho_split_bf16_kernel(const double* __restrict__ phiT, const double* __restrict__ w, int64_t n_grid,
                                      int64_t n_pad, int n_pair, const int* __restrict__ pp,
                                      const int* __restrict__ pq_, int* __restrict__ colexp,
                                      uint16_t* __restrict__ out) {
  const int64_t j = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  const int pq0 = blockIdx.y * 8;
  const int64_t part_stride = static_cast<int64_t>(n_pair) * n_pad;
  for (int u = 0; u < 8; ++u) {
    const int pq = pq0 + u;
    if (pq >= n_pair) break;
    if (j == 0) colexp[pq] = 0;
    if (j >= n_pad) continue;
    const int p = pp[pq], q = pq_[pq];
    const double v = j < n_grid ? w[j] * phiT[p * n_pad + j] * phiT[q * n_pad + j] : 0.0;
    const int64_t o = static_cast<int64_t>(pq) * n_pad + j;
    const __nv_bfloat16 h = __double2bfloat16(v);
    const double r1 = v - static_cast<double>(__bfloat162float(h));
    const __nv_bfloat16 mm = __double2bfloat16(r1);
    const __nv_bfloat16 l = __double2bfloat16(r1 - static_cast<double>(__bfloat162float(mm)));
    out[o] = __bfloat16_as_ushort(h);
    out[part_stride + o] = __bfloat16_as_ushort(mm);
    out[2 * part_stride + o] = __bfloat16_as_ushort(l);
  }
}

// One CTA per row of a step (d) operand: the row maximum sets a power-of-2 scale, then the scaled
// row is split exactly into fp16 hi + lo (simt_pack.cuh), one quantum per accumulation range of 32 KD
// values (`bits` bits).  The source row holds 4 values per outer point (k = 4 i + c); the split row is
// component-major (k' = c * (kdim / 4) + i), so that a range never mixes components.  Lane t holds points 2 t and
// 2 t + 1 of every 64, so that a warp writes whole 128-byte runs of one part.
template <int KD>
__global__ void __launch_bounds__(256) lr_split_kernel(const float* __restrict__ src, int64_t kdim, int bits,
                                                       uint16_t* __restrict__ dst, int* __restrict__ exps,
                                                       uint16_t* __restrict__ dst16) {
  __shared__ float red[8];
  const int64_t r = blockIdx.x;
  const float* s = src + r * kdim;
  float m = 0.0f;
#pragma unroll 4
  for (int64_t k = threadIdx.x * 4; k < kdim; k += blockDim.x * 4) {
    const float4 v = *reinterpret_cast<const float4*>(s + k);
    m = fmaxf(m, fmaxf(fmaxf(fabsf(v.x), fabsf(v.y)), fmaxf(fabsf(v.z), fabsf(v.w))));
  }
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  m = red[0];
  for (int w = 1; w < 8; ++w) m = fmaxf(m, red[w]);
  int e = 0;
  if (m > 0.0f) {
    int em;
    frexpf(m, &em);  // m = f * 2^em, f in [0.5, 1)
    e = min(max(14 - em, -100), 100);
  }
  if (threadIdx.x == 0) exps[r] = e;
  const float scale = ldexpf(1.0f, e);  // exact power of 2 (|e| <= 100)
  uint16_t* d = dst + r * 2 * kdim;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t per_c = kdim / 4;            // outer points, a multiple of 128
  constexpr int G = KD == 4 ? 2 : 1;         // runs of 64 points per step
  for (int64_t i0 = 64 * G * warp; i0 < per_c; i0 += 64 * G * 8) {
    float v[G][2][4];
#pragma unroll
    for (int g = 0; g < G; ++g)
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const float4 q4 = *reinterpret_cast<const float4*>(s + 4 * (i0 + 64 * g + 2 * lane + t));
        v[g][t][0] = q4.x * scale;
        v[g][t][1] = q4.y * scale;
        v[g][t][2] = q4.z * scale;
        v[g][t][3] = q4.w * scale;
      }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float bm = 0.0f;
#pragma unroll
      for (int g = 0; g < G; ++g) bm = fmaxf(bm, fmaxf(fabsf(v[g][0][c]), fabsf(v[g][1][c])));
      bm = __uint_as_float(__reduce_max_sync(KD >= 2 ? 0xffffffffu : (lane < 16 ? 0xffffu : 0xffff0000u), __float_as_uint(bm)));
      const int qe = exact_quantum(bm, bits);
#pragma unroll
      for (int g = 0; g < G; ++g) {
        __half2 h, l;
        split_exact(v[g][0][c], qe, h.x, l.x);
        split_exact(v[g][1][c], qe, h.y, l.y);
        const int64_t kk = c * per_c + i0 + 64 * g;  // first value of the run
        *reinterpret_cast<__half2*>(d + 2 * kk + 2 * lane) = h;
        *reinterpret_cast<__half2*>(d + 2 * kk + 64 + 2 * lane) = l;
        if (dst16)
          *reinterpret_cast<__half2*>(dst16 + r * kdim + kk + 2 * lane) = __floats2half2_rn(v[g][0][c], v[g][1][c]);
      }
    }
  }
}

__global__ void rho_f64_kernel(const double* __restrict__ phi, const double* __restrict__ w, int64_t n_grid,
                               int64_t n_pad, int N, int n_pair, const int* __restrict__ pp,
                               const int* __restrict__ pq_, double* __restrict__ rho) {
  const int64_t j = blockIdx.x;
  for (int pq = blockIdx.y * blockDim.x + threadIdx.x; pq < n_pair; pq += gridDim.y * blockDim.x) {
    double v = 0.0;
    if (j < n_grid) v = w[j] * phi[j * N + pp[pq]] * phi[j * N + pq_[pq]];
    rho[j * n_pair + pq] = v;
  }
}

// ------------------------------------------------------------------ step (a) alone, FP64
__global__ void jastrow_grad_kernel(const JastrowParams* __restrict__ jp, const double* __restrict__ r1,
                                    const double* __restrict__ r2, int64_t n, double* __restrict__ out) {
  const int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (k >= n) return;
  double pc[PT_COEF];
  double nc[MAX_NUC * NUC_COEF];
  double aj[MAX_NUC];
  point_coefs<double>(*jp, r1[3 * k], r1[3 * k + 1], r1[3 * k + 2], 1.0, pc, nc, 0, jp->n_nuc);
  const double x = r2[3 * k], y = r2[3 * k + 1], z = r2[3 * k + 2];
  for (int I = 0; I < jp->n_nuc; ++I) {
    const double dx = x - jp->nuc[I][0], dy = y - jp->nuc[I][1], dz = z - jp->nuc[I][2];
    const double d = sqrt(dx * dx + dy * dy + dz * dz);
    aj[I] = d / (1.0 + d);
  }
  double gx, gy, gz;
  pair_grad_f64(pc, nc, jp->n_nuc, x, y, z, aj, gx, gy, gz);
  out[3 * k] = gx;
  out[3 * k + 1] = gy;
  out[3 * k + 2] = gz;
}

// ------------------------------------------------------------------ steps (a)+(b), FP64 SIMT
// CTA: 32 outer points x 64 pairs x 3 components; K steps of 16 inner points.  The gradient
// tile is generated in shared memory from per-point coefficients (computed once per CTA) and a
// per-inner-point FP64 table (x, y, z, a_jI...).
constexpr int F64_TI = 32, F64_TP = 64, F64_KJ = 16;

__global__ void jtab64_kernel(const double* __restrict__ grid, int64_t n_grid, int64_t n_pad,
                              const JastrowParams* __restrict__ jp, int n_nuc, double* __restrict__ jtab) {
  const int64_t j = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (j >= n_pad) return;
  double x = 1.0e3, y = 1.0e3, z = 1.0e3;
  if (j < n_grid) {
    x = grid[3 * j];
    y = grid[3 * j + 1];
    z = grid[3 * j + 2];
  }
  double* o = jtab + j * (3 + n_nuc);
  o[0] = x;
  o[1] = y;
  o[2] = z;
  for (int I = 0; I < n_nuc; ++I) {
    const double dx = x - jp->nuc[I][0], dy = y - jp->nuc[I][1], dz = z - jp->nuc[I][2];
    const double d = sqrt(dx * dx + dy * dy + dz * dz);
    o[3 + I] = d / (1.0 + d);
  }
}

__global__ void __launch_bounds__(256) vfield_f64_kernel(const double* __restrict__ grid,
                                                          const JastrowParams* __restrict__ jp,
                                                          const double* __restrict__ jtab64,
                                                          const double* __restrict__ rho, int64_t n_pad, int n_pair,
                                                          int64_t i0, int64_t n_i, int64_t gcp,
                                                          const int* __restrict__ pair_p,
                                                          const int* __restrict__ pair_q, int n_orb,
                                                          double* __restrict__ V) {
  extern __shared__ double sm64[];
  const int n_nuc = jp->n_nuc;
  const int cstride = PT_COEF + NUC_COEF * n_nuc;
  double* coef = sm64;                                  // [TI][cstride]
  double* Gs = coef + F64_TI * cstride;                 // [KJ][3][TI]
  double* Rs = Gs + F64_KJ * 3 * F64_TI;                // [KJ][TP]
  const int t = threadIdx.x;
  const int64_t ib = static_cast<int64_t>(blockIdx.x) * F64_TI;
  const int pb = blockIdx.y * F64_TP;
  if (t < F64_TI) {
    const int64_t il = ib + t;
    const int64_t ig = i0 + (il < n_i ? il : n_i - 1);
    double* c = coef + t * cstride;
    point_coefs<double>(*jp, grid[3 * ig], grid[3 * ig + 1], grid[3 * ig + 2], 1.0, c, c + PT_COEF, 0, n_nuc);
  }
  __syncthreads();
  const int tx = t & 31, ty = t >> 5;  // pairs tx, tx+32; points ty*4 .. ty*4+3
  double acc[4][2][3];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int x = 0; x < 3; ++x) acc[a][b][x] = 0.0;
  const int js = 3 + n_nuc;
  for (int64_t j0 = 0; j0 < n_pad; j0 += F64_KJ) {
    for (int k = t; k < F64_KJ * F64_TI; k += 256) {
      const int jj = k / F64_TI, ii = k % F64_TI;
      const double* jr = jtab64 + (j0 + jj) * js;
      const double* c = coef + ii * cstride;
      double gx, gy, gz;
      pair_grad_f64(c, c + PT_COEF, n_nuc, jr[0], jr[1], jr[2], jr + 3, gx, gy, gz);
      Gs[(jj * 3 + 0) * F64_TI + ii] = gx;
      Gs[(jj * 3 + 1) * F64_TI + ii] = gy;
      Gs[(jj * 3 + 2) * F64_TI + ii] = gz;
    }
    for (int k = t; k < F64_KJ * F64_TP; k += 256) {
      const int jj = k / F64_TP, pp = k % F64_TP;
      Rs[k] = (pb + pp < n_pair) ? rho[(j0 + jj) * n_pair + pb + pp] : 0.0;
    }
    __syncthreads();
#pragma unroll 4
    for (int jj = 0; jj < F64_KJ; ++jj) {
      const double r0 = Rs[jj * F64_TP + tx], r1 = Rs[jj * F64_TP + tx + 32];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          const double g = Gs[(jj * 3 + x) * F64_TI + ty * 4 + a];
          acc[a][0][x] = fma(g, r0, acc[a][0][x]);
          acc[a][1][x] = fma(g, r1, acc[a][1][x]);
        }
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int64_t il = ib + ty * 4 + a;
    if (il >= n_i) continue;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int pq = pb + tx + 32 * b;
      if (pq >= n_pair) continue;
      const int p = pair_p[pq], q = pair_q[pq];
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        V[v_index(il, p, q, x, n_orb)] = acc[a][b][x];
        V[v_index(il, q, p, x, n_orb)] = acc[a][b][x];
      }
    }
  }
}

// ------------------------------------------------------------------ final kernels
// In place: M <- Delta U = -(M + M^T) (packed pairs), one CTA per pair of 32 x 32 tiles.
__global__ void symmetrize_kernel(double* __restrict__ M, int n_pair, int ldm) {
  const int bi = blockIdx.y, bj = blockIdx.x;
  if (bj < bi) return;
  __shared__ double A[32][33], B[32][33];
  const int i0 = bi * 32, j0 = bj * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int ri = i0 + r, rj = j0 + r, ci = j0 + threadIdx.x, cj = i0 + threadIdx.x;
    A[r][threadIdx.x] = (ri < n_pair && ci < n_pair) ? M[static_cast<int64_t>(ri) * ldm + ci] : 0.0;
    B[r][threadIdx.x] = (rj < n_pair && cj < n_pair) ? M[static_cast<int64_t>(rj) * ldm + cj] : 0.0;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int ri = i0 + r, ci = j0 + threadIdx.x;
    if (ri < n_pair && ci < n_pair) M[static_cast<int64_t>(ri) * ldm + ci] = -(A[r][threadIdx.x] + B[threadIdx.x][r]);
    const int rj = j0 + r, cj = i0 + threadIdx.x;
    if (bi != bj && rj < n_pair && cj < n_pair)
      M[static_cast<int64_t>(rj) * ldm + cj] = -(B[r][threadIdx.x] + A[threadIdx.x][r]);
  }
}

// dU[p][q][r][s] = U[pair(p,q)][pair(r,s)]: one CTA per (p, q), p <= q, reads its row of U once (the part s < r
// again from L1 / L2) and writes rows (p, q) and (q, p); a warp takes rows r, lanes run over s, so no
// index needs a division.  HBM-bound: 8 (or 4) bytes written per element; one thread per element with two
// divisions took 12.8 ms for N = 200 in FP32 (6.4 GB).
__global__ void __launch_bounds__(256) unpack_kernel(const double* __restrict__ U, int N, int ldm,
                                                     double* __restrict__ dU, float* __restrict__ dU32) {
  const int p = blockIdx.y, q = blockIdx.x;
  if (q < p) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t n2 = static_cast<int64_t>(N) * N;
  const double* src = U + static_cast<int64_t>(pair_of(p, q, N)) * ldm;
  const int64_t o1 = (static_cast<int64_t>(p) * N + q) * n2, o2 = (static_cast<int64_t>(q) * N + p) * n2;
  const bool two = p != q;
  for (int r = warp; r < N; r += 8) {
    const int base_r = r * N - r * (r - 1) / 2 - r;
#pragma unroll 4
    for (int s = lane; s < N; s += 32) {
      const double v = __ldg(src + (s >= r ? base_r + s : s * N - s * (s - 1) / 2 - s + r));
      const int64_t o = static_cast<int64_t>(r) * N + s;
      if (dU) {
        __stcs(dU + o1 + o, v);
        if (two) __stcs(dU + o2 + o, v);
      }
      if (dU32) {
        __stcs(dU32 + o1 + o, static_cast<float>(v));
        if (two) __stcs(dU32 + o2 + o, static_cast<float>(v));
      }
    }
  }
}

// Delta h_pq = -1/2 (2 sum_rs U(pq|rs) gamma_rs - sum_rs U(ps|rq) gamma_rs).  One CTA per row (p, s) of U gives
//   D[ps]      = sum_rt U(ps|rt) gamma_rt   (packed, gpk: gamma_rr, gamma_rt + gamma_tr)
//   Z[p][s][q] = sum_r U(ps|rq) gamma_rs  and  Z[s][p][q] = sum_r U(ps|rq) gamma_rp,
// the latter over the nonzero entries of a column of gamma (lists of gamma_lists_kernel; nothing for an
// empty column), so U is read once, not N^2 gathers per entry of Delta h (16.3 ms for N = 200).  Then
// onebody_sum_kernel adds the columns in order.
__global__ void gamma_lists_kernel(const double* __restrict__ gamma, int N, double* __restrict__ gpk,
                                   int* __restrict__ idx, int* __restrict__ cnt) {
  const int c = blockIdx.x, lane = threadIdx.x;
  int n = 0;
  for (int r0 = 0; r0 < N; r0 += 32) {
    const int r = r0 + lane;
    const double g = r < N ? gamma[r * N + c] : 0.0;
    const unsigned m = __ballot_sync(0xffffffffu, g != 0.0);
    if (g != 0.0) idx[c * N + n + __popc(m & ((1u << lane) - 1))] = r;
    n += __popc(m);
    if (r < c) gpk[pair_of(r, c, N)] = g + gamma[c * N + r];
    if (r == c) gpk[pair_of(r, c, N)] = g;
  }
  if (lane == 0) cnt[c] = n;
}

__device__ __forceinline__ double block_sum_256(double v) {
  __shared__ double red[256];
  red[threadIdx.x] = v;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  return red[0];
}

__global__ void __launch_bounds__(256) onebody_rows_kernel(const double* __restrict__ U, const double* __restrict__ gamma,
                                                           const double* __restrict__ gpk, const int* __restrict__ idx,
                                                           const int* __restrict__ cnt, int N, int NP, int ldm,
                                                           double* __restrict__ D, double* __restrict__ Z) {
  const int p = blockIdx.y, s = blockIdx.x;
  if (s < p) return;
  const int ps = pair_of(p, s, N);
  const double* row = U + static_cast<int64_t>(ps) * ldm;
  double acc = 0.0;
#pragma unroll 4
  for (int k = threadIdx.x; k < NP; k += 256) acc += row[k] * gpk[k];
  const double d = block_sum_256(acc);
  if (threadIdx.x == 0) D[ps] = d;
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    const int a = side ? s : p, c = side ? p : s;   // Z[a][c][.] with column c of gamma
    if (side && p == s) break;
    const int n = cnt[c];
    if (n == 0) continue;
    for (int q = threadIdx.x; q < N; q += 256) {
      double z = 0.0;
      for (int k = 0; k < n; ++k) {
        const int r = idx[c * N + k];
        z += gamma[r * N + c] * row[pair_of(r, q, N)];
      }
      Z[(static_cast<int64_t>(a) * N + c) * N + q] = z;
    }
  }
}

__global__ void onebody_sum_kernel(const double* __restrict__ D, const double* __restrict__ Z,
                                   const int* __restrict__ cnt, int N, double* __restrict__ dh) {
  const int p = blockIdx.y, q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= N) return;
  double x = 0.0;
#pragma unroll 4
  for (int s = 0; s < N; ++s)
    if (cnt[s]) x += Z[(static_cast<int64_t>(p) * N + s) * N + q];
  dh[p * N + q] = -0.5 * (2.0 * D[pair_of(p, q, N)] - x);
}

// Spin builds (Appendix A): U[pq][rs] = -(Fb[pq][rs] + Fa[rs][pq]) = Delta U^{ab}(pq|rs), where
// Ft[pq][rs] = sum_i rho_pq A^t_rs + V_pq.B^t_rs; one CTA per 32 x 32 tile of U.
__global__ void spin_cross_kernel(const double* __restrict__ Fb, const double* __restrict__ Fa, int n_pair, int ldm,
                                  double* __restrict__ U) {
  __shared__ double T[32][33];
  const int i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int ra = j0 + r, ca = i0 + threadIdx.x;  // T[r][x] = Fa[j0 + r][i0 + x]
    T[r][threadIdx.x] = (ra < n_pair && ca < n_pair) ? Fa[static_cast<int64_t>(ra) * ldm + ca] : 0.0;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int row = i0 + r, col = j0 + threadIdx.x;
    if (row < n_pair && col < n_pair)
      U[static_cast<int64_t>(row) * ldm + col] = -(Fb[static_cast<int64_t>(row) * ldm + col] + T[threadIdx.x][r]);
  }
}

// Delta h^s_pq = -1/2 (sum_rs U^{ss}(pq|rs) g^s_rs + sum_rs U^{st}(pq|rs) g^t_rs - sum_rs U^{ss}(ps|rq) g^s_rs),
// t the other spin, U^{ba}(pq|rs) = U^{ab}(rs|pq) (Appendix A); one CTA per (p, q, s).
__global__ void onebody_spin_kernel(const double* __restrict__ Uaa, const double* __restrict__ Uab,
                                    const double* __restrict__ Ubb, const double* __restrict__ ga,
                                    const double* __restrict__ gb, int N, int ldm, double* __restrict__ dh_a,
                                    double* __restrict__ dh_b) {
  const int p = blockIdx.y, q = blockIdx.x, sp = blockIdx.z;
  const double* Us = sp ? Ubb : Uaa;
  const double* gs = sp ? gb : ga;
  const double* go = sp ? ga : gb;
  const int pq = pair_of(p, q, N);
  double acc = 0.0;
  for (int k = threadIdx.x; k < N * N; k += blockDim.x) {
    const int r = k / N, s = k % N;
    const int rs = pair_of(r, s, N);
    const double cross = sp ? Uab[static_cast<int64_t>(rs) * ldm + pq] : Uab[static_cast<int64_t>(pq) * ldm + rs];
    acc += gs[k] * (Us[static_cast<int64_t>(pq) * ldm + rs] -
                    Us[static_cast<int64_t>(pair_of(p, s, N)) * ldm + pair_of(r, q, N)]) +
           go[k] * cross;
  }
  __shared__ double red[256];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) (sp ? dh_b : dh_a)[p * N + q] = -0.5 * red[0];
}

// e0 = -1/3 sum_pq (Delta h^a_pq gamma^a_pq + Delta h^b_pq gamma^b_pq)  (Appendix A)
__global__ void constant_spin_kernel(const double* __restrict__ dh_a, const double* __restrict__ ga,
                                     const double* __restrict__ dh_b, const double* __restrict__ gb, int n2,
                                     double* __restrict__ e0) {
  double acc = 0.0;
  for (int k = threadIdx.x; k < n2; k += blockDim.x) acc += dh_a[k] * ga[k] + dh_b[k] * gb[k];
  __shared__ double red[256];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *e0 = -1.0 / 3.0 * red[0];
}

// e0 = -2/3 sum_pq Delta h_pq gamma_pq
__global__ void __launch_bounds__(1024) constant_kernel(const double* __restrict__ dh, const double* __restrict__ gamma,
                                                        int n2, double* __restrict__ e0) {
  double acc = 0.0;
#pragma unroll 4
  for (int k = threadIdx.x; k < n2; k += blockDim.x) acc += dh[k] * gamma[k];
  __shared__ double red[1024];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *e0 = -2.0 / 3.0 * red[0];
}

template <typename TV>
__global__ void vfield_export_kernel(const TV* __restrict__ V, int splits, int n_pair, int n_orb,
                                     const int* __restrict__ pair_p, const int* __restrict__ pair_q, int64_t n_i,
                                     int64_t gcp, double* __restrict__ out) {
  const int64_t total = n_i * 3 * n_pair;
  const int64_t sstride = v_slice(gcp, n_orb);
  for (int64_t k = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; k < total;
       k += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t pq = k % n_pair, i = k / (3 * n_pair);
    const int x = static_cast<int>((k / n_pair) % 3);
    const int64_t idx = v_index(i, pair_p[pq], pair_q[pq], x, n_orb);
    double v = 0.0;
    for (int z = 0; z < splits; ++z) v += static_cast<double>(V[z * sstride + idx]);
    out[k] = v;
  }
}

inline unsigned int blocks_for(int64_t n, int bs) { return static_cast<unsigned int>((n + bs - 1) / bs); }

}  // namespace

// ------------------------------------------------------------------ launchers
void launch_jtab(const double* grid, int64_t n_grid, int64_t n_pad, const JastrowParams* jp, int n_nuc, int js,
                 float* jtab, cudaStream_t st) {
  jtab_kernel<<<blocks_for(n_pad, 256), 256, 0, st>>>(grid, n_grid, n_pad, jp, n_nuc, js, jtab);
}

void launch_transpose_phi(const double* phi, int64_t n_grid, int64_t n_pad, int N, double* phiT, cudaStream_t st) {
  dim3 grid(blocks_for(n_pad, 32), blocks_for(N, 32));
  transpose_phi_kernel<<<grid, dim3(32, 8), 0, st>>>(phi, n_grid, n_pad, N, phiT);
}

void launch_check_finite(const double* x, int64_t n, int* flag, cudaStream_t st) {
  if (n <= 0) return;
  const unsigned int b = std::min<unsigned int>(blocks_for(n, 256), 4096u);
  check_finite_kernel<<<b, 256, 0, st>>>(x, n, flag);
}

void launch_rho_split(const double* phiT, const double* w, int64_t n_grid, int64_t n_pad, int n_orb, int parts, int kd,
                      const int* pp, const int* pq, unsigned int* colmax, int* colexp, float* phi32, void* out,
                      cudaStream_t st) {
  const int n_pair = n_orb * (n_orb + 1) / 2;
  if (parts == 2) {
    const int64_t total = (static_cast<int64_t>(n_orb) + 1) * n_pad;
    split_phi_f32_kernel<<<std::min<unsigned int>(blocks_for(total, 256), 8192u), 256, 0, st>>>(phiT, w, n_grid,
                                                                                                n_pad, n_orb, phi32);
    cudaMemsetAsync(colmax, 0, sizeof(unsigned int) * n_pair, st);
    rho_colmax_f32_kernel<<<dim3(blocks_for(n_pad, RC_POINTS), n_orb), 256, n_orb * sizeof(unsigned int), st>>>(
        phi32, n_pad, n_orb, colmax);
    rho_colexp_kernel<<<blocks_for(n_pair, 256), 256, 0, st>>>(colmax, n_pair, colexp);
    const dim3 g2(blocks_for(n_pad, RS_POINTS), n_orb);
    uint16_t* o = static_cast<uint16_t*>(out);
    if (kd >= 4)
      rho_split_f16_kernel<4><<<g2, 256, 0, st>>>(phi32, n_pad, n_orb, n_pair, colexp, gemm_bits_b(kd), o);
    else if (kd >= 2)
      rho_split_f16_kernel<2><<<g2, 256, 0, st>>>(phi32, n_pad, n_orb, n_pair, colexp, gemm_bits_b(kd), o);
    else
      rho_split_f16_kernel<1><<<g2, 256, 0, st>>>(phi32, n_pad, n_orb, n_pair, colexp, gemm_bits_b(kd), o);
  } else {
    dim3 g2(blocks_for(n_pad, 256), blocks_for(n_pair, 8));
    rho_split_bf16_kernel<<<g2, 256, 0, st>>>(phiT, w, n_grid, n_pad, n_pair, pp, pq, colexp,
                                               static_cast<uint16_t*>(out));
  }
}

void launch_lr_split(const float* src, int rows, int64_t kdim, int kd, uint16_t* dst, int* exps, uint16_t* dst16,
                     cudaStream_t st) {
  if (rows <= 0) return;
  if (kd >= 4)
    lr_split_kernel<4><<<rows, 256, 0, st>>>(src, kdim, gemm_bits_lr(kd), dst, exps, dst16);
  else if (kd >= 2)
    lr_split_kernel<2><<<rows, 256, 0, st>>>(src, kdim, gemm_bits_lr(kd), dst, exps, dst16);
  else
    lr_split_kernel<1><<<rows, 256, 0, st>>>(src, kdim, gemm_bits_lr(kd), dst, exps, dst16);
}

void launch_rho_f64(const double* phi, const double* w, int64_t n_grid, int64_t n_pad, int n_orb, const int* pp,
                    const int* pq, double* rho, cudaStream_t st) {
  const int n_pair = n_orb * (n_orb + 1) / 2;
  dim3 g(static_cast<unsigned int>(n_pad), std::min<unsigned int>(blocks_for(n_pair, 256), 65535u));
  rho_f64_kernel<<<g, 256, 0, st>>>(phi, w, n_grid, n_pad, n_orb, n_pair, pp, pq, rho);
}

void launch_jastrow_grad(const JastrowParams* jp, const double* r1, const double* r2, int64_t n, double* out,
                         cudaStream_t st) {
  jastrow_grad_kernel<<<blocks_for(n, 64), 64, 0, st>>>(jp, r1, r2, n, out);
}

void launch_jtab64(const double* grid, int64_t n_grid, int64_t n_pad, const JastrowParams* jp, int n_nuc,
                   double* jtab, cudaStream_t st) {
  jtab64_kernel<<<blocks_for(n_pad, 256), 256, 0, st>>>(grid, n_grid, n_pad, jp, n_nuc, jtab);
}

void launch_vfield_f64_impl(const double* grid, const JastrowParams* jp, int n_nuc, const double* jtab64,
                            const double* rho, int64_t n_pad, int n_pair, int64_t i0, int64_t n_i, int64_t gcp,
                            const int* pair_p, const int* pair_q, int n_orb, double* V, cudaStream_t st) {
  const size_t smem = sizeof(double) * (F64_TI * (PT_COEF + NUC_COEF * n_nuc) + F64_KJ * 3 * F64_TI + F64_KJ * F64_TP);
  cudaFuncSetAttribute(vfield_f64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, max_dyn_smem());
  dim3 g(blocks_for(n_i, F64_TI), blocks_for(n_pair, F64_TP));
  vfield_f64_kernel<<<g, 256, smem, st>>>(grid, jp, jtab64, rho, n_pad, n_pair, i0, n_i, gcp, pair_p, pair_q, n_orb,
                                          V);
}

void launch_unpack(const double* M, int n_orb, int n_pair, double* dU, float* dU32, cudaStream_t st) {
  const int ldm = static_cast<int>(m_stride(n_pair));
  if (dU || dU32) {
    unpack_kernel<<<dim3(n_orb, n_orb), 256, 0, st>>>(M, n_orb, ldm, dU, dU32);
  }
}

void launch_symmetrize(double* M, int n_pair, cudaStream_t st) {
  const int ldm = static_cast<int>(m_stride(n_pair));
  dim3 g(blocks_for(n_pair, 32), blocks_for(n_pair, 32));
  symmetrize_kernel<<<g, dim3(32, 8), 0, st>>>(M, n_pair, ldm);
}

size_t onebody_bytes(int n_orb) {
  const size_t n = n_orb, np = n * (n + 1) / 2;
  return 8 * (n * n * n + 2 * np) + 4 * (n * n + n);
}

void launch_onebody(const double* M, const double* gamma, int n_orb, int n_pair, void* tmp, double* dh, double* e0,
                    cudaStream_t st) {
  const int ldm = static_cast<int>(m_stride(n_pair));
  double* Z = static_cast<double*>(tmp);
  double* D = Z + static_cast<size_t>(n_orb) * n_orb * n_orb;
  double* gpk = D + n_pair;
  int* idx = reinterpret_cast<int*>(gpk + n_pair);
  int* cnt = idx + n_orb * n_orb;
  gamma_lists_kernel<<<n_orb, 32, 0, st>>>(gamma, n_orb, gpk, idx, cnt);
  onebody_rows_kernel<<<dim3(n_orb, n_orb), 256, 0, st>>>(M, gamma, gpk, idx, cnt, n_orb, n_pair, ldm, D, Z);
  onebody_sum_kernel<<<dim3(blocks_for(n_orb, 64), n_orb), 64, 0, st>>>(D, Z, cnt, n_orb, dh);
  constant_kernel<<<1, 1024, 0, st>>>(dh, gamma, n_orb * n_orb, e0);
}

void launch_spin_cross(const double* Fb, const double* Fa, int n_pair, double* U, cudaStream_t st) {
  const int ldm = static_cast<int>(m_stride(n_pair));
  dim3 g(blocks_for(n_pair, 32), blocks_for(n_pair, 32));
  spin_cross_kernel<<<g, dim3(32, 8), 0, st>>>(Fb, Fa, n_pair, ldm, U);
}

void launch_onebody_spin(const double* Uaa, const double* Uab, const double* Ubb, const double* ga, const double* gb,
                         int n_orb, int n_pair, double* dh_a, double* dh_b, double* e0, cudaStream_t st) {
  const int ldm = static_cast<int>(m_stride(n_pair));
  onebody_spin_kernel<<<dim3(n_orb, n_orb, 2), 256, 0, st>>>(Uaa, Uab, Ubb, ga, gb, n_orb, ldm, dh_a, dh_b);
  constant_spin_kernel<<<1, 256, 0, st>>>(dh_a, ga, dh_b, gb, n_orb * n_orb, e0);
}

void launch_vfield_export(const void* V, bool f64, int splits, int n_pair, int n_orb, const int* pair_p,
                          const int* pair_q, int64_t n_i, int64_t gcp, double* out, cudaStream_t st) {
  const unsigned int b = std::min<unsigned int>(blocks_for(n_i * 3 * n_pair, 256), 8192u);
  if (f64)
    vfield_export_kernel<double><<<b, 256, 0, st>>>(static_cast<const double*>(V), splits, n_pair, n_orb, pair_p,
                                                    pair_q, n_i, gcp, out);
  else
    vfield_export_kernel<float><<<b, 256, 0, st>>>(static_cast<const float*>(V), splits, n_pair, n_orb, pair_p,
                                                   pair_q, n_i, gcp, out);
}

}  // namespace xtc
