// FP64 contractions on the tensor cores: C[m][n] = sum_k A[m][k] B[n][k] with both operands cut into
// integer digits (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012).
//
// A row of an operand is scaled by a power of 2 (largest magnitude below 2^e) and every value becomes
// x = 2^e sum_d x_d 2^(-8 - 9 d), eight digits of 9 bits, |x_d| <= 2^8, each exact in fp16: 71 bits
// below the row's maximum, against FP64's 53 below each value.  A product of digits i and j belongs to
// diagonal d = i + j; the 36 products with d <= 7 are formed (what is dropped is below 2^-69 of the row
// maxima), all products of one diagonal into one FP32 TMEM accumulator.  Over a range of 64 values of k
// the sums of diagonals 0..3 are integers of at most 2^24 and exact whatever the accumulator's rounding
// (4 x 64 x 2^16 = 2^24); those of diagonals 4..7 would have to line up maximal digits to pass
// 2^24, and a unit of theirs is 2^-36 of the leading one.  After each range the drain warps convert the
// accumulators to integers and add them into two 64-bit integer sums per element, so nothing is
// rounded between the digits and the final conversion to FP64: the order of the sum over k does not
// matter, and the result does not depend on how k is split except for the last FP64 additions.
// In step (b) each inner point j carries a common power of 2 close to w_j max_p phi_p(j)^2 (every orbital
// brought to the same largest value), taken out of rho and multiplied into the pair functions: a row of those is then weighted as in the sum, and its
// maximum is not set by points that contribute nothing (a neighbour of the outer point, a far point
// with no density).  With seven digits and no such scales the error of the water-sized build was 1,500
// times that of the FP64 pipe's sums.  Step (d) uses the same scales for rho and A, others for
// V and B (v_scale_kernel), and the contraction of K those of rho and others for the
// gradients.
//
// Why: the FP64 pipe does 2 FMA per SM and clock on this GPU, the 128 x 32 x 64 FMA of one range of a
// tile take 131,072 of its cycles; the same range is 36 fp16 products of 4 k-steps.  They are bound by shared
// memory, not by the tensor pipe (2,304 cycles): the A planes are read once per k-step (128 KB), the
// stacked B planes 36 / 8 times (144 KB) and the loads write 160 KB, 3,456 cycles at 128 bytes per clock (3,600 measured, the tensor pipe busy
// for 67 to 71 % of them), 36 times the FP64 pipe's rate.  Tile 128 x 32: the eight accumulators take 256 TMEM columns, so that
// two sets fit and the drains of one range overlap the products of the next (64 columns would need
// all 512 and serialise them).
//
// One MMA multiplies digit plane i of A with planes 0..7-i of B stacked as 32 (8 - i) columns (the
// B tile is loaded plane after plane, so its rows are contiguous), and writes diagonals i..7, which
// are adjacent columns of the accumulator set.  Warp 0 loads (A planes through a ring of ten 16 KB
// slots, B tiles through two of 32 KB), warp 1 issues the MMAs, warps 2..9 drain.  Every wait is bounded.
#include <cuda_fp16.h>

#include "digits64.cuh"
#include "gemm_rules.h"
#include "ptx_sm100.cuh"
#include "xtc_internal.cuh"

namespace xtc {
namespace {

constexpr int DIG = D64_PLANES;
constexpr int BM = D64_BM, BN = D64_BN, BK = D64_BK;
constexpr int A_SLOT = BM * BK * 2;             // one digit plane of the A tile: 128 rows of 128 bytes
constexpr int B_SLOT = DIG * BN * BK * 2;       // all digit planes of the B tile
constexpr int A_SLOTS = 10;
constexpr int SMEM = A_SLOTS * A_SLOT + 2 * B_SLOT + 1024 + 256;
constexpr int DRAIN_WARPS = 8;
constexpr int THREADS = (2 + DRAIN_WARPS) * 32;
constexpr int SET_COLS = 256;                   // TMEM columns of an accumulator set
constexpr int HC = BN / 2;                      // columns per drain thread
constexpr int GM = 16;                          // row tiles per group (L2 reuse of the column panels)
static_assert(SMEM <= 232448, "shared memory per CTA");
static_assert(DIG * BN <= SET_COLS && 2 * SET_COLS <= 512, "two accumulator sets in TMEM");
static_assert(DRAIN_WARPS * 32 * HC == BM * BN, "one element of the tile per drain register pair");

__device__ __forceinline__ void tmem_ld_x16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}

// Tile coordinates of CTA L: groups of GM row tiles x every column tile, row fastest.
__device__ __forceinline__ void tile_of(int L, int m_tiles, int n_tiles, int& m, int& n) {
  const int group = L / (GM * n_tiles), first = group * GM;
  const int gm = min(GM, m_tiles - first), rem = L - group * GM * n_tiles;
  m = first + rem % gm;
  n = rem / gm;
}

__global__ void __launch_bounds__(THREADS, 1)
    gemm64_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                  const Gemm64Args args) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* smem_b = smem + A_SLOTS * A_SLOT;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem_b + 2 * B_SLOT);
  uint64_t* a_full = bars;              // [A_SLOTS] the plane landed
  uint64_t* a_free = a_full + A_SLOTS;  // [A_SLOTS] the MMAs of the plane completed
  uint64_t* b_full = a_free + A_SLOTS;  // [2]
  uint64_t* b_free = b_full + 2;        // [2]
  uint64_t* rdone = b_free + 2;         // [2] every MMA of the range in accumulator set b completed
  uint64_t* e_free = rdone + 2;         // [2] the drains released set b
  uint64_t* fin_bar = e_free + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(fin_bar + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  static_assert((2 * A_SLOTS + 9) * 8 + 8 <= 256, "barrier area");

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // warp: uniform
  int m_tile, n_tile;
  tile_of(blockIdx.x, args.m_tiles, args.n_tiles, m_tile, n_tile);
  const int comp = m_tile / args.mt_per_c;
  const int row_c = (m_tile - comp * args.mt_per_c) * BM;               // first row inside the component
  const int row0 = static_cast<int>(comp * args.c_rows) + row_c;
  const int r0 = blockIdx.y * args.ranges_per_split;
  const int n_ranges = min(args.n_ranges, r0 + args.ranges_per_split) - r0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < A_SLOTS; ++s) {
      mbar_init(&a_full[s], 1);
      mbar_init(&a_free[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&b_full[b], 1);
      mbar_init(&b_free[b], 1);
      mbar_init(&rdone[b], 1);
      mbar_init(&e_free[b], DRAIN_WARPS);
    }
    mbar_init(fin_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tm_a);
    tma_prefetch_desc(&tm_b);
  }
  if (warp == 0) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      // ---------------------------------------------------------------- TMA producer
      bool ok = true;
      int a_issued = 0, b_issued = 0;
      for (int r = 0; r < n_ranges && ok; ++r) {
        const int b = r & 1, k0 = (r0 + r) * BK;
        if (r >= 2 && !(ok = mbar_wait(&b_free[b], ((r >> 1) - 1) & 1, abort_flag, args.err, DEV_ERR_TIMEOUT_G64)))
          break;
        mbar_arrive_expect_tx(&b_full[b], B_SLOT);
        tma_load_3d(smem_b + b * B_SLOT, &tm_b, &b_full[b], k0, n_tile * BN, 0);
        b_issued = r + 1;
        for (int i = 0; i < DIG; ++i) {
          const int idx = r * DIG + i, s = idx % A_SLOTS;
          if (idx >= A_SLOTS && !(ok = mbar_wait(&a_free[s], ((idx / A_SLOTS) - 1) & 1, abort_flag, args.err,
                                                 DEV_ERR_TIMEOUT_G64)))
            break;
          mbar_arrive_expect_tx(&a_full[s], A_SLOT);
          tma_load_3d(smem + s * A_SLOT, &tm_a, &a_full[s], k0, row0, i);
          a_issued = idx + 1;
        }
      }
      // the copies still in flight land before the CTA may exit
      int zero = 0;
      volatile int* no_abort = reinterpret_cast<volatile int*>(&zero);
      for (int i = max(0, a_issued - A_SLOTS); i < a_issued; ++i)
        mbar_wait(&a_full[i % A_SLOTS], (i / A_SLOTS) & 1, no_abort, args.err, DEV_ERR_TIMEOUT_G64);
      for (int r = max(0, b_issued - 2); r < b_issued; ++r)
        mbar_wait(&b_full[r & 1], (r >> 1) & 1, no_abort, args.err, DEV_ERR_TIMEOUT_G64);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    // The whole warp, so that descriptors stay in uniform registers; one elected lane issues.  One thread encoding
    // them could not keep up with the pipe: 512 points of a water-sized build (58 orbitals, 40,000 points) 12.7 -> 9.7 ms.
    // The waits vote on every poll, which tells the compiler that the warp stays together: this kernel 5.18 -> 4.64 ms there.
    const uint64_t da0 = sdesc_kmajor_sw128(0) + (smem_u32(smem) >> 4), db0 = sdesc_kmajor_sw128(0) + (smem_u32(smem_b) >> 4);
    const uint32_t a_free_bar = smem_u32(a_free), b_free_bar = smem_u32(b_free), rdone_bar = smem_u32(rdone);
    bool ok = true;
    int s = 0, lap = 0;   // slot of the next A plane and its use
    for (int r = 0; r < n_ranges && ok; ++r) {
      const int b = r & 1, u = r >> 1;
      if (u >= 1 && !(ok = mbar_spin_warp(&e_free[b], (u - 1) & 1, abort_flag, args.err, DEV_ERR_TIMEOUT_G64))) break;
      if (!(ok = mbar_spin_warp(&b_full[b], u & 1, abort_flag, args.err, DEV_ERR_TIMEOUT_G64))) break;
      const uint64_t db = db0 + b * (B_SLOT >> 4);
#pragma unroll
      for (int i = 0; i < DIG; ++i) {
        if (!(ok = mbar_spin_warp(&a_full[s], lap & 1, abort_flag, args.err, DEV_ERR_TIMEOUT_G64))) break;
        tc_fence_after();
        const uint64_t da = da0 + s * (A_SLOT >> 4);
        const uint32_t d = tmem + b * SET_COLS + i * BN;
#pragma unroll
        for (int k = 0; k < BK / 16; ++k)  // 16 values = 32 bytes = 2 descriptor units
          tc_mma_f16_warp(d, da + 2 * k, db + 2 * k, idesc_f16(BM, BN * (DIG - i), false), (i | k) ? 1u : 0u);
        tc_commit_warp(a_free_bar + 8 * s);
        if (++s == A_SLOTS) {
          s = 0;
          ++lap;
        }
      }
      if (!ok) break;
      tc_commit_warp(b_free_bar + 8 * b);
      tc_commit_warp(rdone_bar + 8 * b);
    }
    tc_commit_warp(smem_u32(fin_bar));
    int zero = 0;
    mbar_wait(fin_bar, 0, reinterpret_cast<volatile int*>(&zero), args.err, DEV_ERR_TIMEOUT_G64);
  } else {
    // ------------------------------------------------------------------ drains and epilogue
    const int quarter = warp & 3;               // TMEM lanes 32*quarter .. +31 (hardware rule)
    const int col0 = ((warp - 2) >> 2) * HC;
    const uint32_t base = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + col0;
    // element = 2^(e_a + e_b - 43) (hi + lo 2^-36): diagonals 0..3 in hi, 4..7 in lo
    long long hi[HC], lo[HC];
#pragma unroll
    for (int c = 0; c < HC; ++c) hi[c] = lo[c] = 0;
    bool ok = true;
    for (int r = 0; r < n_ranges; ++r) {
      const int b = r & 1;
      ok = mbar_spin_warp(&rdone[b], (r >> 1) & 1, abort_flag, args.err, DEV_ERR_TIMEOUT_G64);
      if (!ok) break;
      tc_fence_after();
      const uint32_t src = base + b * SET_COLS;
      // two diagonals at a time
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        uint32_t e0[HC], e1[HC];
        tmem_ld_x16(src + 2 * h * BN, e0);
        tmem_ld_x16(src + (2 * h + 1) * BN, e1);
        tmem_wait_ld();
        if (h == 3) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&e_free[b]);
        }
#pragma unroll
        for (int c = 0; c < HC; ++c) {
          long long& acc = h < 2 ? hi[c] : lo[c];
          acc += static_cast<long long>(__float2int_rn(__uint_as_float(e0[c]))) * (h & 1 ? 1 << 9 : 1 << 27);
          acc += static_cast<long long>(__float2int_rn(__uint_as_float(e1[c]))) * (h & 1 ? 1 : 1 << 18);
        }
      }
    }
    if (ok) {
      const int row = quarter * 32 + lane;
      const int ea = row_c + row < args.m_rows ? __ldg(args.exp_a + row0 + row) : 0;
      double* out = args.C + (static_cast<int64_t>(blockIdx.y) * gridDim.x + blockIdx.x) * (BM * BN) + row;
#pragma unroll
      for (int c = 0; c < HC; ++c) {
        const int col = n_tile * BN + col0 + c;
        const int eb = col < args.n_cols ? __ldg(args.exp_b + col) : 0;
        double v = fma(static_cast<double>(lo[c]), 0x1p-36, static_cast<double>(hi[c]));
        v = scalbn(v, ea + eb - 43);
        if (max(ea, eb) >= D64_NONFINITE) v = __longlong_as_double(0x7ff8000000000000ll);
        out[(col0 + c) * BM] = v;
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ------------------------------------------------------------------ what becomes of the tiles
// One CTA per tile and four columns (thread = row): the sum of the slices of k in order, then
//   TO_V     V[v_index(i, p, s, x)] of both (p, s) and (s, p) (component = x, row = point i, column = pair)
//   TO_ROWS  out[pair][((c0 + component) mod 4) * ld_c + i]
//   ADD      out[row][column] += value (row stride ld)
// With o.add the first two add to what is there (a further block of inner points).
enum { TO_V = 0, TO_ROWS = 1, ADD = 2 };
template <int MODE>
__global__ void __launch_bounds__(BM) gemm64_finalize_kernel(const Gemm64Args a, int splits, const Gemm64Out o) {
  int m_tile, n_tile;
  tile_of(blockIdx.x, a.m_tiles, a.n_tiles, m_tile, n_tile);
  const int comp = m_tile / a.mt_per_c;
  const int64_t row = static_cast<int64_t>(m_tile - comp * a.mt_per_c) * BM + threadIdx.x;
  if (row >= a.m_rows) return;
  const double* src = a.C + static_cast<int64_t>(blockIdx.x) * (BM * BN) + (blockIdx.y * 4) * BM + threadIdx.x;
  const int64_t zs = static_cast<int64_t>(gridDim.x) * (BM * BN);
  double v[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
  for (int z = 0; z < splits; ++z)
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] += src[z * zs + c * BM];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int col = n_tile * BN + blockIdx.y * 4 + c;
    if (col >= a.n_cols) return;
    if (MODE == TO_V) {
      const int p = __ldg(o.pair_p + col), s = __ldg(o.pair_q + col);
      double* dst = o.out + v_index(o.i0 + row, p, s, comp, o.n_orb);
      if (o.add) v[c] += *dst;
      *dst = v[c];
      o.out[v_index(o.i0 + row, s, p, comp, o.n_orb)] = v[c];
    } else if (MODE == TO_ROWS) {
      double* dst = o.out + col * o.ld + ((o.c0 + comp) & 3) * o.ld_c + o.i0 + row;
      *dst = o.add ? *dst + v[c] : v[c];
    } else {
      o.out[row * o.ld + col] += v[c];
    }
  }
}

// ------------------------------------------------------------------ digits of an operand
constexpr int DG_THREADS = 256;

// The digits are relative to a row's maximum, so each source also gives the power of 2 that its values
// at index k carry (and the other operand's do not): with s_j, the point scale, rho is of order 2^s_j at
// point j, and what it multiplies is weighted by it.

// Operand of step (d) from FP64 rows, k = 4 i + c: L = (rho, V) and R = (A, B).  Both parts of L go without their scales
// (sign -1), sj for rho and sv for V (v_scale_kernel), which bring them to the heights of the pair's orbitals, and
// those of R with them (sign +1).  With rho alone scaled, V kept what bits its size beside phi^2 left it: none of the
// result's was right with weights of 1e-40 (sums of w phi^2 are 1 for orthonormal orbitals, but no input has to be).
struct LrSrc {
  static constexpr bool GROUPED = true;
  const double* p;
  int64_t ld, k0;           // first k of the block
  const int* sj;            // of the chunk's first point
  const int* sv;
  int64_t n_i;
  int sign;
  // four values from k on, k a multiple of 4: one point's
  __device__ void load4(int64_t row, int64_t k, double (&v)[4], int (&s)[4]) const {
    const double2* q = reinterpret_cast<const double2*>(p + row * ld + k);
    const double2 a = q[0], b = q[1];
    v[0] = a.x;
    v[1] = a.y;
    v[2] = b.x;
    v[3] = b.y;
    const int64_t i = (k0 + k) >> 2;
    const int j = i < n_i ? sj[i] : 0, g = i < n_i ? sv[i] : 0;
    s[0] = j <= D64_NO_SCALE ? D64_NO_SCALE : sign * j;
    s[1] = s[2] = s[3] = g <= D64_NO_SCALE ? D64_NO_SCALE : sign * g;
  }
};
// rho^T[pq][j] = w_j phi_p(j) phi_q(j), times 2^-sj[j]
struct RhoSrc {
  static constexpr bool GROUPED = false;
  const double* phiT;
  int64_t ld;
  const double* w;
  const int* pair_p;
  const int* pair_q;
  const int* sj;
  __device__ double at(int64_t row, int64_t k) const {
    return w[k] * phiT[pair_p[row] * ld + k] * phiT[pair_q[row] * ld + k];
  }
  __device__ int scale(int64_t k) const { return sj[k] == D64_NO_SCALE ? D64_NO_SCALE : -sj[k]; }
};
// Operands of the contraction of K, k = c ncp + i, i < n_i a point of the chunk (zero past them).  Left: row
// pq = p N + q, c = 0: w phi_p phi_q / 2, c = 1..3: w phi_p d_x phi_q (dphiT row 3 q + x).  Right: W, V_x.  W grows as 1/r
// next to a nucleus, where the weight is as small, and gradients have a length in them, so both kinds of k carry scales of their
// own, sj (as in step (b)) and sg (point_scale_kernel), taken out of the left operand and multiplied into the right one.
// Without any a point 1e-12 bohr from a nucleus cost every row the bits of 1/r, 1e-10 of max |K| where FP64 sums give
// 1e-14; with one for both, a grid 1e-12 bohr across did.
__device__ __forceinline__ int k_component(int64_t k, int64_t ncp) { return (k >= ncp) + (k >= 2 * ncp) + (k >= 3 * ncp); }
struct PsiSrc {
  static constexpr bool GROUPED = false;
  const double* phiT;
  const double* dphiT;
  int64_t ld;
  const double* w;
  const int* sj;
  const int* sg;
  int64_t i0, n_i, ncp;
  int n_orb;
  __device__ double at(int64_t row, int64_t k) const {
    const int c = k_component(k, ncp);
    const int64_t i = k - c * ncp, g = i0 + i;
    if (i >= n_i) return 0.0;
    const int64_t p = row / n_orb, q = row - p * n_orb;
    const double wp = w[g] * phiT[p * ld + g];
    return c == 0 ? 0.5 * wp * phiT[q * ld + g] : wp * dphiT[(3 * q + c - 1) * ld + g];
  }
  __device__ int scale(int64_t k) const {
    const int c = k_component(k, ncp);
    const int64_t i = k - c * ncp, g = i0 + i;
    if (i >= n_i) return 0;
    const int s = c ? sg[g] : sj[g];
    return s == D64_NO_SCALE ? D64_NO_SCALE : -s;
  }
};
struct WvSrc {
  static constexpr bool GROUPED = true;
  const double* p;
  const int* sj;
  const int* sg;
  int64_t i0, n_i, ncp;
  __device__ void load4(int64_t row, int64_t k, double (&v)[4], int (&s)[4]) const {
    const double2* q = reinterpret_cast<const double2*>(p + row * 4 * ncp + k);
    const double2 a = q[0], b = q[1];
    v[0] = a.x;
    v[1] = a.y;
    v[2] = b.x;
    v[3] = b.y;
    const int c = k_component(k, ncp);   // of all four: ncp is a multiple of 64
    const int64_t i = k - c * ncp;
    const int* sc = (c ? sg : sj) + i0 + i;
#pragma unroll
    for (int t = 0; t < 4; ++t) s[t] = i + t < n_i ? sc[t] : 0;
  }
};

// One CTA per row: the row's largest exponent, then the digits of four consecutive k per thread.  The
// digits come out of the bit pattern with integer operations (the FP64 pipe is the scarce one): two
// passes over the row, the second from L2.
template <class Src>
__global__ void __launch_bounds__(DG_THREADS) digits_kernel(const Src src, int64_t K, int64_t Kp,
                                                            uint16_t* __restrict__ planes, int64_t plane,
                                                            int* __restrict__ exps) {
  const int64_t row = blockIdx.x;
  int m = 0;
  if constexpr (Src::GROUPED) {   // K is a multiple of 4
#pragma unroll 2
    for (int64_t k = 4 * threadIdx.x; k < K; k += 4 * DG_THREADS) {
      double v[4];
      int s[4];
      src.load4(row, k, v, s);
#pragma unroll
      for (int t = 0; t < 4; ++t) m = max(m, d64_key(v[t], s[t]));
    }
  } else {
    for (int64_t k = threadIdx.x; k < K; k += DG_THREADS) m = max(m, d64_key(src.at(row, k), src.scale(k)));
  }
  __shared__ int red[32];
  const int e = d64_exponent(block_max(m, red));
  if (threadIdx.x == 0) exps[row] = e;
  uint16_t* out = planes + row * Kp;
  for (int64_t k = 4 * threadIdx.x; k < Kp; k += 4 * DG_THREADS) {
    double v[4];
    int s[4];
    if constexpr (Src::GROUPED) {
      src.load4(row, k, v, s);
    } else {
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        v[t] = k + t < K ? src.at(row, k + t) : 0.0;
        s[t] = k + t < K ? src.scale(k + t) : 0;
      }
    }
    d64_store_digits(v, s, e, out + k, plane);
  }
}

// orb[p] (initially 0): the largest key of row p over the grid, OK_POINTS points a CTA.
constexpr int OK_POINTS = 8 * DG_THREADS;
__global__ void __launch_bounds__(DG_THREADS) orbital_key_kernel(const double* __restrict__ phiT, int64_t ld,
                                                                 int64_t n_grid, int* __restrict__ orb) {
  __shared__ int red[32];
  const int64_t j0 = static_cast<int64_t>(blockIdx.x) * OK_POINTS + threadIdx.x;
  double v[OK_POINTS / DG_THREADS];
#pragma unroll
  for (int t = 0; t < OK_POINTS / DG_THREADS; ++t) {
    const int64_t j = j0 + t * DG_THREADS;
    v[t] = j < n_grid ? phiT[blockIdx.y * ld + j] : 0.0;
  }
  int m = 0;
#pragma unroll
  for (int t = 0; t < OK_POINTS / DG_THREADS; ++t) m = max(m, d64_key(v[t], 0));
  m = block_max(m, red);
  if (threadIdx.x == 0 && m) atomicMax(orb + blockIdx.y, m);
}

// sj[j]: the exponent of |w_j| max_p (phi_p(j) / max phi_p)^2, the largest pair product of inner point j with
// every orbital brought to the same height; D64_NO_SCALE where that is 0 (every pair product is 0 then).  With dphiT, sg[j]
// instead: |w_j| max_p (|phi_p(j)| / max |phi_p|) max_q,x (|d_x phi_q(j)| / max |phi_q|), for the operands of K (an orbital
// that is 0 everywhere: at the height of its gradient).  orb[n_orb], dorb[3 n_orb]: largest keys of the orbitals and of their
// gradients.  Latency-bound: PS_GROUPS threads share a point's orbitals.
constexpr int PS_GROUPS = 8;
__global__ void __launch_bounds__(32 * PS_GROUPS)
    point_scale_kernel(const double* __restrict__ phiT, const double* __restrict__ dphiT, int64_t ld,
                       const double* __restrict__ w, int64_t n_j, int n_orb, const int* __restrict__ orb,
                       const int* __restrict__ dorb, int* __restrict__ sj) {
  __shared__ int red[2][PS_GROUPS][32];
  const int64_t j = blockIdx.x * 32ll + threadIdx.x;
  int m = D64_NO_SCALE, mg = D64_NO_SCALE;
  if (j < n_j) {
#pragma unroll 2
    for (int p = threadIdx.y; p < n_orb; p += PS_GROUPS) {
      const int k = d64_key(phiT[p * ld + j], 0);
      if (k) m = max(m, k - orb[p]);
      if (dphiT) {
        int kd = 0, top = 0;
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          kd = max(kd, d64_key(dphiT[(3 * p + x) * ld + j], 0));
          top = max(top, dorb[3 * p + x]);
        }
        if (kd) mg = max(mg, kd - (orb[p] ? orb[p] : top));
      }
    }
  }
  red[0][threadIdx.y][threadIdx.x] = m;
  red[1][threadIdx.y][threadIdx.x] = mg;
  __syncthreads();
  if (threadIdx.y || j >= n_j) return;
#pragma unroll
  for (int g = 1; g < PS_GROUPS; ++g) {
    m = max(m, red[0][g][threadIdx.x]);
    mg = max(mg, red[1][g][threadIdx.x]);
  }
  if (!dphiT) mg = m;
  const int kw = d64_key(w[j], 0);
  sj[j] = m == D64_NO_SCALE || mg == D64_NO_SCALE || kw == 0 ? D64_NO_SCALE : kw - D64_BIAS - 1022 + m + mg;
}

// sv[i], initially below D64_NO_SCALE: the exponent of max_pq,x |V_x,pq(i)| / (max phi_p max phi_q), from the rows of L; stays
// below where V is 0.  One thread per point and VS_PAIRS pairs.
constexpr int VS_PAIRS = 8;
__global__ void __launch_bounds__(128) v_scale_kernel(const double* __restrict__ L, int64_t ld, int64_t n_i, int n_pair,
                                                      const int* __restrict__ pair_p, const int* __restrict__ pair_q,
                                                      const int* __restrict__ orb, int* __restrict__ sv) {
  __shared__ int height[VS_PAIRS];
  const int64_t i = blockIdx.x * 128ll + threadIdx.x;
  const int pq0 = blockIdx.y * VS_PAIRS, pq1 = min(n_pair, pq0 + VS_PAIRS);
  if (pq0 + threadIdx.x < pq1) height[threadIdx.x] = orb[pair_p[pq0 + threadIdx.x]] + orb[pair_q[pq0 + threadIdx.x]];
  __syncthreads();
  if (i >= n_i) return;
  int m = D64_NO_SCALE;
  double2 v[VS_PAIRS][2];   // all in flight
#pragma unroll
  for (int t = 0; t < VS_PAIRS; ++t) {
    const double2* p = reinterpret_cast<const double2*>(L + static_cast<int64_t>(min(pq0 + t, n_pair - 1)) * ld + 4 * i);
    v[t][0] = p[0];
    v[t][1] = p[1];
  }
#pragma unroll
  for (int t = 0; t < VS_PAIRS; ++t) {
    const int k = max(d64_key(v[t][0].y, 0), max(d64_key(v[t][1].x, 0), d64_key(v[t][1].y, 0)));
    if (pq0 + t < pq1 && k && k < D64_NONFINITE) m = max(m, k - height[t] + D64_BIAS + 1022);
  }
  if (m > D64_NO_SCALE) atomicMax(sv + i, m);
}

}  // namespace

size_t gemm64_tile_bytes(int m_tiles, int n_tiles, int splits) {
  return static_cast<size_t>(m_tiles) * n_tiles * splits * BM * BN * sizeof(double);
}

void launch_gemm64(const CUtensorMap* tm_a, const CUtensorMap* tm_b, const Gemm64Args& in, int splits,
                   cudaStream_t st) {
  if (in.m_tiles <= 0 || in.n_tiles <= 0 || in.n_ranges <= 0) return;
  Gemm64Args a = in;
  a.ranges_per_split = (a.n_ranges + splits - 1) / splits;
  cudaFuncSetAttribute(gemm64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
  gemm64_kernel<<<dim3(static_cast<unsigned>(a.m_tiles * a.n_tiles), static_cast<unsigned>(splits)), THREADS, SMEM,
                  st>>>(*tm_a, *tm_b, a);
}

void launch_gemm64_finalize(const Gemm64Args& a, int splits, const Gemm64Out& o, int mode, cudaStream_t st) {
  if (a.m_tiles <= 0 || a.n_tiles <= 0) return;
  const dim3 g(static_cast<unsigned>(a.m_tiles * a.n_tiles), BN / 4);
  if (mode == D64_TO_V)
    gemm64_finalize_kernel<TO_V><<<g, BM, 0, st>>>(a, splits, o);
  else if (mode == D64_TO_ROWS)
    gemm64_finalize_kernel<TO_ROWS><<<g, BM, 0, st>>>(a, splits, o);
  else
    gemm64_finalize_kernel<ADD><<<g, BM, 0, st>>>(a, splits, o);
}

void launch_v_scale(const double* L, int64_t ld, int64_t n_i, int n_pair, const int* pair_p, const int* pair_q,
                    const int* orb, int* sv, cudaStream_t st) {
  cudaMemsetAsync(sv, 0x80, n_i * sizeof(int), st);   // below D64_NO_SCALE
  v_scale_kernel<<<dim3(static_cast<unsigned>((n_i + 127) / 128), static_cast<unsigned>((n_pair + VS_PAIRS - 1) / VS_PAIRS)), 128,
                   0, st>>>(L, ld, n_i, n_pair, pair_p, pair_q, orb, sv);
}

void launch_digits_lr(const double* src, int64_t rows, int64_t ld, int64_t k0, int64_t K, const int* sj, const int* sv,
                      int64_t n_i, int sign, uint16_t* planes, int* exps, cudaStream_t st) {
  if (rows <= 0) return;
  digits_kernel<<<static_cast<unsigned>(rows), DG_THREADS, 0, st>>>(LrSrc{src + k0, ld, k0, sj, sv, n_i, sign}, K, K,
                                                                    planes, rows * K, exps);
}

void launch_digits_rho(const double* phiT, int64_t ld, const double* w, int64_t n_j, int64_t Kp, int n_orb,
                       const int* pair_p, const int* pair_q, const int* sj, uint16_t* planes, int* exps,
                       cudaStream_t st) {
  const int64_t rows = static_cast<int64_t>(n_orb) * (n_orb + 1) / 2;
  digits_kernel<<<static_cast<unsigned>(rows), DG_THREADS, 0, st>>>(RhoSrc{phiT, ld, w, pair_p, pair_q, sj}, n_j, Kp,
                                                                    planes, rows * Kp, exps);
}

void launch_point_scale(const double* phiT, int64_t ld, const double* w, int64_t n_grid, int n_orb, int* orb, int* sj,
                        cudaStream_t st) {
  cudaMemsetAsync(orb, 0, n_orb * sizeof(int), st);
  orbital_key_kernel<<<dim3(static_cast<unsigned>((n_grid + OK_POINTS - 1) / OK_POINTS), n_orb), DG_THREADS, 0, st>>>(
      phiT, ld, n_grid, orb);
  point_scale_kernel<<<static_cast<unsigned>((n_grid + 31) / 32), dim3(32, PS_GROUPS), 0, st>>>(phiT, nullptr, ld, w, n_grid,
                                                                                             n_orb, orb, nullptr, sj);
}

void launch_gradient_scale(const double* phiT, const double* dphiT, int64_t ld, const double* w, int64_t n_grid,
                           int n_orb, const int* orb, int* dorb, int* sg, cudaStream_t st) {
  cudaMemsetAsync(dorb, 0, 3 * n_orb * sizeof(int), st);
  orbital_key_kernel<<<dim3(static_cast<unsigned>((n_grid + OK_POINTS - 1) / OK_POINTS), 3 * n_orb), DG_THREADS, 0, st>>>(
      dphiT, ld, n_grid, dorb);
  point_scale_kernel<<<static_cast<unsigned>((n_grid + 31) / 32), dim3(32, PS_GROUPS), 0, st>>>(phiT, dphiT, ld, w, n_grid,
                                                                                             n_orb, orb, dorb, sg);
}

void launch_digits_psi(const double* phiT, const double* dphiT, int64_t ld, const double* w, const int* sj, const int* sg,
                       int64_t i0, int64_t n_i, int64_t ncp, int n_orb, uint16_t* planes, int* exps, cudaStream_t st) {
  const int64_t rows = static_cast<int64_t>(n_orb) * n_orb;
  digits_kernel<<<static_cast<unsigned>(rows), DG_THREADS, 0, st>>>(
      PsiSrc{phiT, dphiT, ld, w, sj, sg, i0, n_i, ncp, n_orb}, 4 * ncp, 4 * ncp, planes, rows * 4 * ncp, exps);
}

void launch_digits_wv(const double* src, int64_t rows, const int* sj, const int* sg, int64_t i0, int64_t n_i, int64_t ncp,
                      uint16_t* planes, int* exps, cudaStream_t st) {
  digits_kernel<<<static_cast<unsigned>(rows), DG_THREADS, 0, st>>>(WvSrc{src, sj, sg, i0, n_i, ncp}, 4 * ncp, 4 * ncp,
                                                                    planes, rows * 4 * ncp, exps);
}

}  // namespace xtc
