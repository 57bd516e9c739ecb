// Step (a) in FP64 for the tensor-core contraction (gemm64_tc.cu): the Jastrow gradient
// G_x(i, j) = d/dx_i u(r_i, r_j) of every (outer point i, inner point j) pair of a chunk and, for the
// two-body integrals K, F(i, j) = lap_1 u + |grad_1 u|^2, written as digit rows.
//
// u = sum_I sum_t c (a1^m a2^n + a1^n a2^m) b^o with a = r/(1+r) for the electron-nucleus distances and b
// the same for r12 (jastrow_coef.cuh).  With the first electron's factors taken into coefficients,
//   grad_1 u = E + H b' e12,   E = K0 + b K1 + b^2 K2 + sum_I a2 t_I(a2, b) g_I,   H = h1 + b h2 = du/db,
//   lap_1 u  = L0 + b L1 + b^2 L2 + h2 b'^2 + 2 H b' (1/r12 - 1/(1+r12)) + 2 b' e12 . dE/db,
// where L_o holds a'^2 d2/da1^2 + (a'' + 2 a'/r1) d/da1 of the terms in b^o (a polynomial in a2 per
// nucleus), b' = (1 + r12)^-2, b'' = -2 b'/(1 + r12).  A zero-length unit vector (a point on a nucleus,
// r12 = 0) and the 1/r terms that go with it contribute zero; everything else is kept.
//
// Bound by the FP64 pipe (2 instructions per SM and clock): about 60 FP64 instructions a pair for the
// gradient with two nuclei, 100 with F, where summing F term by term took ten times that.  So 1/r12
// and 1/(1+r12) come from the FP32 approximations by one third-order step (error of the step below
// 2^-60, then FP64 rounding), conversions and digits are integer operations on bit patterns, and the
// values are formed once per pair, not once per tile of orbital pairs.  A CTA takes one outer point at
// a time: the row in FP64 into its scratch row (L2) with the row maximum, then the digits.
#include <algorithm>

#include "digits64.cuh"
#include "jastrow_coef.cuh"
#include "simt_pack.cuh"
#include "xtc_internal.cuh"

namespace xtc {
namespace {

constexpr int THREADS = 256;
constexpr int CTAS_PER_SM = 3;
constexpr double EPS2 = 1e-28;   // (1e-14 bohr)^2

// Coefficients of one outer point in shared memory, scalars first, then one record per nucleus.
struct PointCoef {
  double x, y, z;
  double K[3][3];     // k = 0 parts of E: [o][x]
  double Hc1, Hc2;    // k = 0 parts of H
  double L[3];        // k = 0 parts of L_o
};
struct NucCoef {
  double g[3];
  double a01, a02, a11, a12, a21, a22;   // derivative with respect to a1: [o][k] for k >= 1
  double b11, b12, b21, b22;             // o times the term: [o][k] for k >= 1
  double L[3][2];                        // [o][k - 1]
  double al0[3], be0[2], L0[3];          // k = 0 parts, summed over nuclei into PointCoef
};

__device__ __forceinline__ void nuc_coef(const JastrowParams& jp, int I, double x, double y, double z, NucCoef& q) {
  const double vx = x - jp.nuc[I][0], vy = y - jp.nuc[I][1], vz = z - jp.nuc[I][2];
  const double d = sqrt(vx * vx + vy * vy + vz * vz);
  const double s1 = 1.0 / (1.0 + d), a1 = d * s1, ap = s1 * s1;
  const double inv = d < 1e-14 ? 0.0 : 1.0 / d;
  const double radial = -2.0 * ap * s1 + 2.0 * ap * inv;  // a'' + 2 a'/r
  q.g[0] = vx * (ap * inv);
  q.g[1] = vy * (ap * inv);
  q.g[2] = vz * (ap * inv);
  double al[3][3], be[3][3], dd[3][3];
#pragma unroll
  for (int o = 0; o < 3; ++o)
#pragma unroll
    for (int k = 0; k < 3; ++k) al[o][k] = be[o][k] = dd[o][k] = 0.0;
  const double pw[3] = {1.0, a1, a1 * a1};
  const int set = jp.set[I];
  for (int t = 0; t < jp.n_terms; ++t) {
    const int m = jp.mno[t][0], n = jp.mno[t][1], o = jp.mno[t][2];
    const double c = jp.coef[set][t];
#pragma unroll
    for (int sw = 0; sw < 2; ++sw) {
      const int p1 = sw ? n : m, p2 = sw ? m : n;   // a1^p1 a2^p2
      const double v = c * pw[p1], d1 = p1 ? c * p1 * pw[p1 - 1] : 0.0, d2 = p1 == 2 ? 2.0 * c : 0.0;
#pragma unroll
      for (int oo = 0; oo < 3; ++oo)
#pragma unroll
        for (int k = 0; k < 3; ++k)
          if (oo == o && k == p2) {
            al[oo][k] += d1;
            be[oo][k] += oo * v;
            dd[oo][k] += d2;
          }
    }
  }
  q.a01 = al[0][1];
  q.a02 = al[0][2];
  q.a11 = al[1][1];
  q.a12 = al[1][2];
  q.a21 = al[2][1];
  q.a22 = al[2][2];
  q.b11 = be[1][1];
  q.b12 = be[1][2];
  q.b21 = be[2][1];
  q.b22 = be[2][2];
  q.be0[0] = be[1][0];
  q.be0[1] = be[2][0];
#pragma unroll
  for (int o = 0; o < 3; ++o) {
    q.al0[o] = al[o][0];
    q.L0[o] = ap * ap * dd[o][0] + radial * al[o][0];
    q.L[o][0] = ap * ap * dd[o][1] + radial * al[o][1];
    q.L[o][1] = ap * ap * dd[o][2] + radial * al[o][2];
  }
}

// FP32 value of a normal FP64 number in [2^-126, 2^127) (truncated) and back (exact), by the bit patterns.
__device__ __forceinline__ float narrow(double x) {
  return __uint_as_float(__funnelshift_l(static_cast<uint32_t>(__double2loint(x)),
                                         static_cast<uint32_t>(__double2hiint(x)) - (896u << 20), 3));
}
__device__ __forceinline__ double widen(float y) {
  const uint32_t b = __float_as_uint(y);
  return __hiloint2double(static_cast<int>((b >> 3) + (896u << 20)), static_cast<int>(b << 29));
}
// 1/sqrt(x), x > 0: y0 + y0 e (1/2 + 3/8 e) with e = 1 - x y0^2 (third order).
__device__ __forceinline__ double rsqrt64(double x) {
  if (!(x > 1e-36 && x < 1e36)) return 1.0 / sqrt(x);
  const double y = widen(rsqrt_approx(narrow(x)));
  const double e = fma(-(x * y), y, 1.0);
  return fma(fma(0.375, e, 0.5), e * y, y);
}
// 1/x, x >= 1: y0 + y0 (e + e^2) with e = 1 - x y0.
__device__ __forceinline__ double rcp64(double x) {
  if (!(x < 1e36)) return 1.0 / x;
  const double y = widen(rcp_approx(narrow(x)));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

template <int NC>
__global__ void __launch_bounds__(THREADS, CTAS_PER_SM)
    grad64_kernel(const double* __restrict__ grid, const JastrowParams* __restrict__ jp, int n_nuc,
                  const double* __restrict__ jt, const int* __restrict__ sj, int64_t ld, int64_t n_j, int64_t Kp,
                  int64_t i0, int64_t n_i, int64_t c_rows, double* __restrict__ scratch, uint16_t* __restrict__ planes, int64_t plane,
                  int* __restrict__ exps) {
  constexpr bool GRAD = NC >= 3, LAP = NC == 1 || NC == 4;
  extern __shared__ __align__(16) uint8_t smem_raw[];
  __shared__ PointCoef pt;
  __shared__ int red[32];
  NucCoef* nuc = reinterpret_cast<NucCoef*>(smem_raw);
  double* rows = scratch + static_cast<int64_t>(blockIdx.x) * NC * Kp;
  for (int64_t il = blockIdx.x; il < n_i; il += gridDim.x) {
    const double px = grid[3 * (i0 + il)], py = grid[3 * (i0 + il) + 1], pz = grid[3 * (i0 + il) + 2];
    __syncthreads();  // the previous point's coefficients and rows are no longer read
    for (int I = threadIdx.x; I < n_nuc; I += THREADS) nuc_coef(*jp, I, px, py, pz, nuc[I]);
    __syncthreads();
    if (threadIdx.x < 14) {
      // thread k sums one k = 0 coefficient over the nuclei in order
      const int k = threadIdx.x;
      double s = 0.0;
      for (int I = 0; I < n_nuc; ++I) {
        const NucCoef& q = nuc[I];
        s += k < 9 ? q.al0[k / 3] * q.g[k % 3] : (k < 11 ? q.be0[k - 9] : q.L0[k - 11]);
      }
      (k < 9 ? pt.K[k / 3][k % 3] : (k == 9 ? pt.Hc1 : (k == 10 ? pt.Hc2 : pt.L[k - 11]))) = s;
    }
    __syncthreads();
    // ------------------------------------------------------------ the row in FP64, and its largest exponents
    int mx[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) mx[c] = 0;
    for (int64_t j = threadIdx.x; j < n_j; j += THREADS) {
      const double dx = px - __ldg(jt + j), dy = py - __ldg(jt + ld + j), dz = pz - __ldg(jt + 2 * ld + j);
      const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
      const double i12 = r2 > EPS2 ? rsqrt64(r2) : 0.0;
      // below 1e-14 bohr the distance still enters b (the unit vector does not)
      const double r = r2 > EPS2 ? r2 * i12 : sqrt(r2);
      const double s12 = rcp64(1.0 + r);
      const double b = r * s12, bp = s12 * s12;
      double ex = fma(b, fma(b, pt.K[2][0], pt.K[1][0]), pt.K[0][0]);
      double ey = fma(b, fma(b, pt.K[2][1], pt.K[1][1]), pt.K[0][1]);
      double ez = fma(b, fma(b, pt.K[2][2], pt.K[1][2]), pt.K[0][2]);
      double h1 = pt.Hc1, h2 = pt.Hc2;
      double fx = 0.0, fy = 0.0, fz = 0.0, l0 = 0.0, l1 = 0.0, l2 = 0.0;
      if (LAP) {
        const double b2 = b + b;
        fx = fma(b2, pt.K[2][0], pt.K[1][0]);
        fy = fma(b2, pt.K[2][1], pt.K[1][1]);
        fz = fma(b2, pt.K[2][2], pt.K[1][2]);
        l0 = pt.L[0];
        l1 = pt.L[1];
        l2 = pt.L[2];
      }
      for (int I = 0; I < n_nuc; ++I) {
        const NucCoef& q = nuc[I];
        const double a = __ldg(jt + (3 + I) * ld + j);
        const double u1 = fma(a, q.a12, q.a11), u2 = b * fma(a, q.a22, q.a21);
        const double at = a * fma(b, u1 + u2, fma(a, q.a02, q.a01));
        ex = fma(at, q.g[0], ex);
        ey = fma(at, q.g[1], ey);
        ez = fma(at, q.g[2], ez);
        h1 = fma(a, fma(a, q.b12, q.b11), h1);
        h2 = fma(a, fma(a, q.b22, q.b21), h2);
        if (LAP) {
          const double ad = a * fma(2.0, u2, u1);
          fx = fma(ad, q.g[0], fx);
          fy = fma(ad, q.g[1], fy);
          fz = fma(ad, q.g[2], fz);
          l0 = fma(a, fma(a, q.L[0][1], q.L[0][0]), l0);
          l1 = fma(a, fma(a, q.L[1][1], q.L[1][0]), l1);
          l2 = fma(a, fma(a, q.L[2][1], q.L[2][0]), l2);
        }
      }
      const double h = fma(b, h2, h1);
      const double s = bp * i12, hs = h * s;   // b' e12 = s d
      const double gx = fma(hs, dx, ex), gy = fma(hs, dy, ey), gz = fma(hs, dz, ez);
      double v[4] = {gx, gy, gz, 0.0};
      if (LAP) {
        double f = fma(b, fma(b, l2, l1), l0);
        f = fma(h2 * bp, bp, f);
        f = fma(2.0 * (h * bp), i12 - s12, f);
        f = fma(2.0 * s, fma(dx, fx, fma(dy, fy, dz * fz)), f);
        f = fma(gx, gx, fma(gy, gy, fma(gz, gz, f)));
        v[NC == 1 ? 0 : 3] = f;
      }
      const int s_j = __ldg(sj + j);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        rows[c * Kp + j] = v[c];
        mx[c] = max(mx[c], d64_key(v[c], s_j));
      }
    }
    // ------------------------------------------------------------ digits of the rows
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const int e = d64_exponent(block_max(mx[c], red));  // the barriers also publish the FP64 row
      const int64_t row = (GRAD ? c : 0) * c_rows + il;
      if (threadIdx.x == 0) exps[row] = e;
      for (int64_t k = 4 * threadIdx.x; k < Kp; k += 4 * THREADS) {
        double v[4];
        int s[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          v[t] = k + t < n_j ? rows[c * Kp + k + t] : 0.0;
          s[t] = k + t < n_j ? __ldg(sj + k + t) : 0;
        }
        d64_store_digits(v, s, e, planes + row * Kp + k, plane);
      }
    }
  }
}

__global__ void jtab64_soa_kernel(const double* __restrict__ grid, int64_t n_grid, int64_t n_pad,
                                  const JastrowParams* __restrict__ jp, int n_nuc, double* __restrict__ jt) {
  const int64_t j = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (j >= n_pad) return;
  double x = 1.0e3, y = 1.0e3, z = 1.0e3;
  if (j < n_grid) {
    x = grid[3 * j];
    y = grid[3 * j + 1];
    z = grid[3 * j + 2];
  }
  jt[j] = x;
  jt[n_pad + j] = y;
  jt[2 * n_pad + j] = z;
  for (int I = 0; I < n_nuc; ++I) {
    const double dx = x - jp->nuc[I][0], dy = y - jp->nuc[I][1], dz = z - jp->nuc[I][2];
    const double d = sqrt(dx * dx + dy * dy + dz * dz);
    jt[(3 + I) * n_pad + j] = d / (1.0 + d);
  }
}

unsigned grad_ctas(int64_t n_i, int n_sm) {
  return static_cast<unsigned>(std::min<int64_t>(n_i, static_cast<int64_t>(n_sm) * CTAS_PER_SM));
}

}  // namespace

size_t grad64_scratch_bytes(int comps, int64_t n_i, int64_t Kp, int n_sm) {
  return static_cast<size_t>(grad_ctas(n_i, n_sm)) * comps * Kp * sizeof(double);
}

void launch_jtab64_soa(const double* grid, int64_t n_grid, int64_t n_pad, const JastrowParams* jp, int n_nuc,
                       double* jt, cudaStream_t st) {
  jtab64_soa_kernel<<<static_cast<unsigned>((n_pad + 127) / 128), 128, 0, st>>>(grid, n_grid, n_pad, jp, n_nuc, jt);
}

void launch_grad64_digits(const double* grid, const JastrowParams* jp, int n_nuc, const double* jt, const int* sj,
                          int64_t ld, int64_t n_j, int64_t Kp, int64_t i0, int64_t n_i, int64_t c_rows, int comps, double* scratch,
                          uint16_t* planes, int* exps, int n_sm, cudaStream_t st) {
  if (n_i <= 0) return;
  const unsigned ctas = grad_ctas(n_i, n_sm);
  const size_t smem = sizeof(NucCoef) * n_nuc;   // at most 64 nuclei: 14 KB
  const int64_t plane = comps * c_rows * Kp;
  if (comps == 3)
    grad64_kernel<3><<<ctas, THREADS, smem, st>>>(grid, jp, n_nuc, jt, sj, ld, n_j, Kp, i0, n_i, c_rows, scratch, planes,
                                                  plane, exps);
  else if (comps == 4)
    grad64_kernel<4><<<ctas, THREADS, smem, st>>>(grid, jp, n_nuc, jt, sj, ld, n_j, Kp, i0, n_i, c_rows, scratch, planes,
                                                  plane, exps);
  else
    grad64_kernel<1><<<ctas, THREADS, smem, st>>>(grid, jp, n_nuc, jt, sj, ld, n_j, Kp, i0, n_i, c_rows, scratch, planes,
                                                  plane, exps);
}

}  // namespace xtc
