// Step (a) in FP64 for the tensor-core contraction (gemm64_tc.cu): the Jastrow gradient
// G_x(i, j) = d/dx_i u(r_i, r_j) of every (outer point i, inner point j) pair of a chunk and, for the
// two-body integrals K, F(i, j) = lap_1 u + |grad_1 u|^2, written as digit rows.
//
// u = sum_I sum_t c (a1^m a2^n + a1^n a2^m) b^o with a = r/(1+r) for the electron-nucleus distances and b
// the same for r12 (jastrow_coef.cuh).  With the first electron's factors taken into coefficients,
//   grad_1 u = E + H b' e12,   E = K0 + b K1 + b^2 K2 + sum_I a2 t_I(a2, b) g_I,   H = h1 + b h2 = du/db,
//   lap_1 u  = L0 + b L1 + b^2 L2 + h2 b'^2 + 2 H b' (1/r12 - 1/(1+r12)) + 2 b' e12 . dE/db
//            = L0 + b L1 + b^2 L2 + 3 h2 b'^2 + 2 h1 b' / (r12 (1+r12)) + 2 b' e12 . dE/db,
// (b (1/r12 - 1/(1+r12)) = b'; so 1/r12 meets h1 alone, which has a scale of its own and is exactly 0 where du/db
// vanishes at r12 = 0: with H / r12 from one fixed-point H a pair 1e-7 bohr apart lost 1e-11 of F with terms in b^2 only)
// where L_o holds a'^2 d2/da1^2 + (a'' + 2 a'/r1) d/da1 of the terms in b^o (a polynomial in a2 per
// nucleus), b' = (1 + r12)^-2, b'' = -2 b'/(1 + r12).  A zero-length unit vector (a point on a nucleus,
// r12 = 0) and the 1/r terms that go with it contribute zero; everything else is kept.
//
// Bound by the FP64 pipe (2 instructions per SM and clock; with every term in FP64 130 instructions a pair for F
// with three nuclei).  The polynomials in a2 and b, nine tenths of the arithmetic, have arguments in
// [0, 1) and coefficients that are fixed for an outer point, so they are evaluated in 64-bit fixed point on the
// integer pipe: coefficients scaled per outer point so that the sum of all magnitudes stays below 2^59 to 2^61, products
// rounded to units of that scale, 2^-59 of that sum or less, where FP64 rounds every term to 2^-53 of itself.  What is left in FP64 are the distances, b' and the last products, about 35 instructions.
// 1/r12 and 1/(1+r12) come from the FP32 approximations by one third-order step (error of the step below
// 2^-60, then FP64 rounding), comparisons, conversions and digits are integer operations on bit patterns, and the
// values are formed once per pair, not once per tile of orbital pairs.  A CTA takes one outer point at
// a time: the row in FP64 into its scratch row (L2) with the row maximum, then the digits.
// Calls, all FP64 -> fixed point (one GB300): K with 30 orbitals, 8,000 points and 3 nuclei 18.8 -> 10.6 ms, K on an H2-sized input
// 1,168 -> 770 us, its FP64 build 847 -> 659 us, 512 points of a water-sized build 9.7 -> 8.3 ms.  Rows that it does not
// resolve are evaluated in FP64 (BITS_GRAD), so the errors against 64 bits are those of the FP64 pipe; with that check, the
// scale of its own for h1 and the points' scales of K and V those calls take 10.6 ms, 834 us, 680 us and (with the waits
// of gemm64_tc.cu) 7.8 ms.
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

// ------------------------------------------------------------------ fixed point
// Scale of coefficients whose magnitudes do not add up to a finite number (infinities, NaN, sums beyond the FP64
// range): what is evaluated from them is NaN (from_fixed_rare, which every value of such a scale goes through).
constexpr int NO_RANGE = 1 << 20;
// x 2^s as an integer, rounded to nearest (|x| 2^s < 2^63).
__device__ __forceinline__ long long to_fixed(double x, int s) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
  const int ex = static_cast<int>(b >> 52) & 0x7ff;
  const unsigned long long m = (b & 0xfffffffffffffull) | (ex ? 1ull << 52 : 0ull);
  const int sh = max(ex, 1) - 1075 + s;
  const unsigned long long u = sh >= 0 ? m << min(sh, 63) : (sh > -55 ? (m + (1ull << (-sh - 1))) >> -sh : 0ull);
  return static_cast<long long>(b) < 0 ? -static_cast<long long>(u) : static_cast<long long>(u);
}
// A factor t as t_h 2^32 + t_l with both halves signed 32-bit (|t_l| <= 2^31), so that a product takes three signed
// 32 x 32 multiplications; packed as (t_h, t_l).
__device__ __forceinline__ long long halves(long long t) {
  const int l = static_cast<int>(t);
  const unsigned h = static_cast<unsigned>(t >> 32) + (static_cast<unsigned>(l) >> 31);
  return static_cast<long long>((static_cast<unsigned long long>(h) << 32) | static_cast<unsigned>(l));
}
// x t / 2^(64 - UP) for |x|, |t| < 2^62 (t in halves), rounded; the product of the low halves is left out (at most
// 2^(UP - 2) units, either sign).
template <int UP>
__device__ __forceinline__ long long mulh(long long x, long long t) {
  const long long xb = halves(x);
  const long long xh = static_cast<int>(xb >> 32), xl = static_cast<int>(xb), th = static_cast<int>(t >> 32), tl = static_cast<int>(t);
  return xh * th * (1 << UP) + ((xh * tl + xl * th + (1ll << (31 - UP))) >> (32 - UP));
}
// x in [0, 1] as x 2^62, truncated, in halves.
__device__ __forceinline__ long long unit_fixed(double x) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
  const int sh = static_cast<int>(b >> 52) - 1013;   // at most 10
  const unsigned long long m = (b & 0xfffffffffffffull) | (1ull << 52);
  return halves(static_cast<long long>(sh >= 0 ? m << min(sh, 10) : m >> min(-sh, 63)));
}
// The rare forms out of line: inlined they are predicated, and their FP64 instructions issue for every pair (45 of
// 81 a pair before).
__device__ __noinline__ double from_fixed_rare(long long v, int s) {
  return s == NO_RANGE ? __longlong_as_double(0x7ff8000000000000ll) : scalbn(static_cast<double>(v), -s);
}
__device__ __noinline__ double sqrt_rare(double x) { return sqrt(x); }
__device__ __noinline__ double rsqrt_rare(double x) { return 1.0 / sqrt(x); }
__device__ __noinline__ double rcp_rare(double x) { return 1.0 / x; }
// v 2^-s in FP64, rounded to nearest.
__device__ __forceinline__ double from_fixed(long long v, int s) {
  const unsigned long long u = v < 0 ? 0ull - static_cast<unsigned long long>(v) : static_cast<unsigned long long>(v);
  const int lz = __clzll(static_cast<long long>(u));
  const int ex = 1085 - lz - s;   // biased exponent less one
  if (static_cast<unsigned>(ex) > 2044u) return from_fixed_rare(v, s);
  const unsigned long long m = u << (lz & 63);
  const unsigned long long r = (static_cast<unsigned long long>(ex) << 52) + (m >> 11) + ((m >> 10) & 1);
  return u ? __longlong_as_double(static_cast<long long>(r | (static_cast<unsigned long long>(v) & 0x8000000000000000ull)))
           : 0.0;
}
// x t, t a fraction from unit_fixed.
__device__ __forceinline__ long long mulf(long long x, long long t) { return mulh<2>(x, t); }
// Exponent e with |x| < 2^e (x finite); 0 for 0, so that sums of no terms stay clear of the rare forms.
__device__ __forceinline__ int exponent_above(double x) {
  return x == 0.0 ? 0 : max(static_cast<int>((__double_as_longlong(x) >> 52) & 0x7ff), 1) - 1022;
}

// The fixed-point coefficients of an outer point.  Scales: a.. of nucleus I by 2^(61 - e_I), e_I bounding the sum of their
// magnitudes; g of nucleus I so that their products, and K, carry 2^sE; b1. and Hc1 2^sH1, b2. and Hc2 2^sH2 (one scale
// where F is not asked for), L 2^sL.
struct NucFix {
  long long a01, a02, a11, a12, a21, a22, g[3];
  long long b11, b12, b21, b22;
  long long L[3][2];
};
struct PointFix {
  long long K[3][3], Hc1, Hc2, L[3];
  int sE, sH1, sH2, sL;
  int uE, uH1, uH2, uL;   // exponents of their units; NO_UNIT where the sum is empty, and exact
};
__device__ __forceinline__ double bound_a(const NucCoef& q) {
  return fabs(q.a01) + fabs(q.a02) + fabs(q.a11) + fabs(q.a12) + 2.0 * (fabs(q.a21) + fabs(q.a22));
}
__device__ __forceinline__ int scale_of(double sum, int bits) {
  return sum < INFINITY ? bits - exponent_above(sum) : NO_RANGE;   // NaN is not below
}
constexpr int NO_UNIT = -(1 << 20);
__device__ __forceinline__ int unit_of(double sum, int scale) { return sum == 0.0 ? NO_UNIT : -scale; }
// The larger of two magnitudes, NaN if either is (fmax would drop it).
__device__ __forceinline__ double nan_max(double a, double b) { return b <= a ? a : (a <= b ? b : a + b); }
// Threads 0, 1, 2: the scales of E, H and L.
template <bool LAP>
__device__ __forceinline__ void point_scales(const PointCoef& pt, const NucCoef* nuc, int n_nuc, int k, PointFix& f) {
  double s = 0.0, s2 = 0.0, s3 = 0.0;
  if (k == 0) {
    for (int x = 0; x < 3; ++x) s = nan_max(s, fabs(pt.K[0][x]) + fabs(pt.K[1][x]) + 2.0 * fabs(pt.K[2][x]));
    for (int I = 0; I < n_nuc; ++I)
      s += bound_a(nuc[I]) * nan_max(fabs(nuc[I].g[0]), nan_max(fabs(nuc[I].g[1]), fabs(nuc[I].g[2])));
    f.sE = scale_of(s, 61);
    f.uE = unit_of(s, f.sE);
  } else if (k == 1) {
    s = fabs(pt.Hc1);
    s2 = fabs(pt.Hc2);
    for (int I = 0; I < n_nuc; ++I) {
      s += fabs(nuc[I].b11) + fabs(nuc[I].b12);
      s2 += fabs(nuc[I].b21) + fabs(nuc[I].b22);
    }
    if (!LAP) s = s2 = nan_max(s, s2);
    f.sH1 = scale_of(s, 60);
    f.sH2 = scale_of(s2, 60);
    f.uH1 = unit_of(s, f.sH1);
    f.uH2 = unit_of(s2, f.sH2);
  } else {
    s = fabs(pt.L[0]);
    s2 = fabs(pt.L[1]);
    s3 = fabs(pt.L[2]);
    for (int I = 0; I < n_nuc; ++I) {
      s += fabs(nuc[I].L[0][0]) + fabs(nuc[I].L[0][1]);
      s2 += fabs(nuc[I].L[1][0]) + fabs(nuc[I].L[1][1]);
      s3 += fabs(nuc[I].L[2][0]) + fabs(nuc[I].L[2][1]);
    }
    s = nan_max(s, nan_max(s2, s3));
    f.sL = scale_of(s, 59);
    f.uL = unit_of(s, f.sL);
  }
}
__device__ __forceinline__ void nuc_fix(const NucCoef& q, const PointFix& p, NucFix& f) {
  const int eI = exponent_above(bound_a(q)), sa = 61 - eI, sg = p.sE + eI;  // at g / 2^61 then carries sE
  f.a01 = to_fixed(q.a01, sa);
  f.a02 = to_fixed(q.a02, sa);
  f.a11 = to_fixed(q.a11, sa);
  f.a12 = to_fixed(q.a12, sa);
  f.a21 = to_fixed(q.a21, sa);
  f.a22 = to_fixed(q.a22, sa);
  for (int x = 0; x < 3; ++x) f.g[x] = halves(to_fixed(q.g[x], sg));
  f.b11 = to_fixed(q.b11, p.sH1);
  f.b12 = to_fixed(q.b12, p.sH1);
  f.b21 = to_fixed(q.b21, p.sH2);
  f.b22 = to_fixed(q.b22, p.sH2);
  for (int o = 0; o < 3; ++o)
    for (int k = 0; k < 2; ++k) f.L[o][k] = to_fixed(q.L[o][k], p.sL);
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
  if (static_cast<unsigned>((__double2hiint(x) >> 20) - 904) > 238u) return rsqrt_rare(x);   // outside 2^-119 .. 2^120
  const double y = widen(rsqrt_approx(narrow(x)));
  const double e = fma(-(x * y), y, 1.0);
  return fma(fma(0.375, e, 0.5), e * y, y);
}
// 1/x, x >= 1: y0 + y0 (e + e^2) with e = 1 - x y0.
__device__ __forceinline__ double rcp64(double x) {
  if (static_cast<unsigned>(__double2hiint(x) >> 20) > 1142u) return rcp_rare(x);
  const double y = widen(rcp_approx(narrow(x)));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// Exponent e with x < 2^e for x >= 0 of the given high word.
__device__ __forceinline__ int exponent_of_hi(int hi) { return (hi >> 20) - 1022; }

// Largest values of the CTA for M values a thread, to every thread; scratch: M ints a warp.
template <int M>
__device__ __forceinline__ void block_max_n(int* v, int* scratch) {
  constexpr int W = THREADS / 32;
#pragma unroll
  for (int c = 0; c < M; ++c) v[c] = __reduce_max_sync(0xffffffffu, v[c]);
  __syncthreads();
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int c = 0; c < M; ++c) scratch[c * W + (threadIdx.x >> 5)] = v[c];
  __syncthreads();
#pragma unroll
  for (int c = 0; c < M; ++c)
#pragma unroll
    for (int w = 0; w < W; ++w) v[c] = max(v[c], scratch[c * W + w]);
}

// The pair functions in FP64 throughout, for rows that the fixed point does not resolve: v[0..2] the gradient, v[3] F.
__device__ __forceinline__ void pair_fp64(const JastrowParams& jp, const PointCoef& pt, const NucCoef* nuc, double dx,
                                       double dy, double dz, double xj, double yj, double zj, double (&v)[4]) {
  const double r2 = dx * dx + dy * dy + dz * dz, r = sqrt(r2);
  const bool apart = r2 > EPS2;
  const double i12 = apart ? 1.0 / r : 0.0, s12 = 1.0 / (1.0 + r), b = r * s12, bp = s12 * s12, s = bp * i12;
  double e[3], fe[3], h1 = pt.Hc1, h2 = pt.Hc2, l[3] = {pt.L[0], pt.L[1], pt.L[2]};
#pragma unroll
  for (int x = 0; x < 3; ++x) {
    e[x] = pt.K[0][x] + b * (pt.K[1][x] + b * pt.K[2][x]);
    fe[x] = pt.K[1][x] + 2.0 * b * pt.K[2][x];
  }
  for (int I = 0; I < jp.n_nuc; ++I) {
    const NucCoef& q = nuc[I];
    const double ux = xj - jp.nuc[I][0], uy = yj - jp.nuc[I][1], uz = zj - jp.nuc[I][2];
    const double d = sqrt(ux * ux + uy * uy + uz * uz), a = d / (1.0 + d);
    const double u1 = q.a11 + q.a12 * a, u2 = (q.a21 + q.a22 * a) * b;
    const double at = a * (q.a01 + q.a02 * a + b * (u1 + u2)), ad = a * (u1 + 2.0 * u2);
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      e[x] += at * q.g[x];
      fe[x] += ad * q.g[x];
      l[x] += a * (q.L[x][0] + q.L[x][1] * a);
    }
    h1 += a * (q.b11 + q.b12 * a);
    h2 += a * (q.b21 + q.b22 * a);
  }
  const double h = h1 + b * h2, hs = h * s;
  v[0] = hs * dx + e[0];
  v[1] = hs * dy + e[1];
  v[2] = hs * dz + e[2];
  const double t = s * (dx * fe[0] + dy * fe[1] + dz * fe[2]) + (apart ? h1 * s : -(h * bp)) * s12;
  v[3] = l[0] + b * (l[1] + b * l[2]) + (apart ? 3.0 : 1.0) * (h2 * bp) * bp + 2.0 * t + v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
}

// This thread's part of a row, and its largest exponents.
template <int NC>
__device__ __noinline__ void row_fp64(const JastrowParams& jp, const PointCoef& pt, const NucCoef* nuc, double px,
                                      double py, double pz, const double* jt, int64_t ld, int64_t n_j, int64_t Kp,
                                      const int* sj, double* rows, int* mx) {
  for (int c = 0; c < NC; ++c) mx[c] = 0;
  for (int64_t j = threadIdx.x; j < n_j; j += THREADS) {
    const double xj = jt[j], yj = jt[ld + j], zj = jt[2 * ld + j];
    double v[4];
    pair_fp64(jp, pt, nuc, px - xj, py - yj, pz - zj, xj, yj, zj, v);
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      rows[c * Kp + j] = v[NC == 1 ? 3 : c];
      mx[c] = max(mx[c], d64_key(v[NC == 1 ? 3 : c], sj[j]));
    }
  }
}

// Bits that the largest entry of a row (with its points' scales) has to stand above the largest error unit of the fixed point
// for the row to be kept; else it is evaluated again in FP64.  Rows of molecules stand 54 and more above it
// (gradient) and 47 and more (F, whose unit is bounded less closely: far outer points).  Rows below are those of
// outer points whose coefficients meet only small powers of a2 or b where the weight is: grids far smaller than a bohr,
// densities within 1e-6 bohr of a nucleus.  They lost up to half of their bits.
constexpr int BITS_GRAD = 50, BITS_F = 46;

// Does the row of largest key `key` stand less than `bits` above the unit 2^unit (some error, not infinite or NaN)?
__device__ __forceinline__ bool short_of(int key, int unit, int bits) {
  return unit > NO_UNIT / 2 && key < D64_NONFINITE && (key == 0 || key - D64_BIAS - 1022 - unit < bits);
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
  __shared__ int red[(NC + 1) * (THREADS / 32)];
  __shared__ PointFix pf;
  NucCoef* nuc = reinterpret_cast<NucCoef*>(smem_raw);
  NucFix* nf = reinterpret_cast<NucFix*>(nuc + n_nuc);
  double* rows = scratch + static_cast<int64_t>(blockIdx.x) * NC * Kp;
  int s_max = 2 * NO_UNIT;   // the largest point scale
  for (int64_t j = threadIdx.x; j < n_j; j += THREADS) s_max = max(s_max, __ldg(sj + j));
  block_max_n<1>(&s_max, red);
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
    if (threadIdx.x < 3) point_scales<LAP>(pt, nuc, n_nuc, threadIdx.x, pf);
    __syncthreads();
    for (int I = threadIdx.x; I < n_nuc; I += THREADS) nuc_fix(nuc[I], pf, nf[I]);
    if (threadIdx.x < 14) {
      const int k = threadIdx.x;
      if (k < 9)
        pf.K[k / 3][k % 3] = to_fixed(pt.K[k / 3][k % 3], pf.sE);
      else if (k < 11)
        (k == 9 ? pf.Hc1 : pf.Hc2) = to_fixed(k == 9 ? pt.Hc1 : pt.Hc2, k == 9 ? pf.sH1 : pf.sH2);
      else
        pf.L[k - 11] = to_fixed(pt.L[k - 11], pf.sL);
    }
    __syncthreads();
    const int sE = pf.sE, sH1 = pf.sH1, sH2 = pf.sH2, sL = pf.sL;
    // ------------------------------------------------------------ the row in FP64, and its largest exponents
    int mx[NC + 1];   // and of b' max(1, 1/r12 if F is asked for) with the points' scales
#pragma unroll
    for (int c = 0; c < NC; ++c) mx[c] = 0;
    mx[NC] = 2 * NO_UNIT;
    for (int64_t j = threadIdx.x; j < n_j; j += THREADS) {
      const double dx = px - __ldg(jt + j), dy = py - __ldg(jt + ld + j), dz = pz - __ldg(jt + 2 * ld + j);
      const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
      const bool apart = __double_as_longlong(r2) > __double_as_longlong(EPS2);   // r2 > EPS2
      const double i12 = apart ? rsqrt64(r2) : 0.0;
      // below 1e-14 bohr the distance still enters b (the unit vector does not)
      const double r = apart ? r2 * i12 : sqrt_rare(r2);
      const double s12 = rcp64(1.0 + r);
      const double b = r * s12, bp = s12 * s12;
      const long long B = unit_fixed(b);
      long long e[3], fe[3];   // E and dE/db
#pragma unroll
      for (int x = 0; x < 3; ++x) {
        const long long kb = mulf(pf.K[2][x], B);
        e[x] = pf.K[0][x] + mulf(pf.K[1][x] + kb, B);
        fe[x] = pf.K[1][x] + 2 * kb;
      }
      long long h1 = pf.Hc1, h2 = pf.Hc2, l0 = pf.L[0], l1 = pf.L[1], l2 = pf.L[2];
      for (int I = 0; I < n_nuc; ++I) {
        const NucFix& q = nf[I];
        const long long A = __ldg(reinterpret_cast<const long long*>(jt) + (3 + I) * ld + j);   // a2
        const long long u1 = q.a11 + mulf(q.a12, A), u2 = mulf(q.a21 + mulf(q.a22, A), B);
        const long long at = mulf(q.a01 + mulf(q.a02, A) + mulf(u1 + u2, B), A);
#pragma unroll
        for (int x = 0; x < 3; ++x) e[x] += mulh<3>(at, q.g[x]);
        h1 += mulf(q.b11 + mulf(q.b12, A), A);
        h2 += mulf(q.b21 + mulf(q.b22, A), A);
        if (LAP) {
          const long long ad = mulf(u1 + 2 * u2, A);
#pragma unroll
          for (int x = 0; x < 3; ++x) fe[x] += mulh<3>(ad, q.g[x]);
          l0 += mulf(q.L[0][0] + mulf(q.L[0][1], A), A);
          l1 += mulf(q.L[1][0] + mulf(q.L[1][1], A), A);
          l2 += mulf(q.L[2][0] + mulf(q.L[2][1], A), A);
        }
      }
      const double h1d = LAP ? from_fixed(h1, sH1) : 0.0;
      const double h = LAP ? fma(b, from_fixed(h2, sH2), h1d) : from_fixed(h1 + mulf(h2, B), sH1);
      const double s = bp * i12, hs = h * s;   // b' e12 = s d
      const double gx = fma(hs, dx, from_fixed(e[0], sE)), gy = fma(hs, dy, from_fixed(e[1], sE)),
                   gz = fma(hs, dz, from_fixed(e[2], sE));
      double v[4] = {gx, gy, gz, 0.0};
      if (LAP) {
        const double fx = from_fixed(fe[0], sE), fy = from_fixed(fe[1], sE), fz = from_fixed(fe[2], sE);
        double f = from_fixed(l0 + mulf(l1 + mulf(l2, B), B), sL);
        // where 1/r12 counts as 0: h2 b'^2 - 2 H b' / (1+r12)
        f = fma(from_fixed(apart ? 3 * h2 : h2, sH2) * bp, bp, f);
        const double t = fma(s, fma(dx, fx, fma(dy, fy, dz * fz)), (apart ? h1d * s : -(h * bp)) * s12);
        f = fma(2.0, t, f);
        f = fma(gx, gx, fma(gy, gy, fma(gz, gz, f)));
        v[NC == 1 ? 0 : 3] = f;
      }
      const int s_j = __ldg(sj + j);
      mx[NC] = max(mx[NC], s_j + exponent_of_hi(LAP ? max(__double2hiint(s), __double2hiint(bp)) : __double2hiint(bp)));
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        rows[c * Kp + j] = v[c];
        mx[c] = max(mx[c], d64_key(v[c], s_j));
      }
    }
    block_max_n<NC + 1>(mx, red);  // the barriers also publish the FP64 row
    // the largest error unit of the row: of the gradient max(2^uE, b' 2^uH), of F also (the gradient's) times twice the gradient,
    // and h1's times b' / r12
    const int uE = pf.uE, uH = max(pf.uH1, pf.uH2), top = max(max(uE + 61, uH + 60) + 1, 0);
    bool again = false;
    if (GRAD) again = short_of(max(mx[0], max(mx[1], mx[2])), max(s_max + uE, mx[NC] + uH), BITS_GRAD);
    if (LAP) again |= short_of(mx[NC - 1], max(s_max + max(pf.uL, uE + top + 1), mx[NC] + uH + top + 2), BITS_F);
    if (again) {   // the same for all threads
      int m[NC];
      row_fp64<NC>(*jp, pt, nuc, px, py, pz, jt, ld, n_j, Kp, sj, rows, m);
      block_max_n<NC>(m, red);
#pragma unroll
      for (int c = 0; c < NC; ++c) mx[c] = m[c];
    }
    // ------------------------------------------------------------ digits of the rows
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      const int e = d64_exponent(mx[c]);
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
    reinterpret_cast<long long*>(jt)[(3 + I) * n_pad + j] = unit_fixed(d / (1.0 + d));
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
  const size_t smem = (sizeof(NucCoef) + sizeof(NucFix)) * n_nuc;   // at most 64 nuclei: 24 KB
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
