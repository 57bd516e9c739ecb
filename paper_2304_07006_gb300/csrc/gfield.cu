// Step (a) for the tensor-core path: the Jastrow gradient G_x(i, j) = d/dx_i u(r_i, r_j) of every
// (outer point i, inner point j) pair of a chunk (section "Decomposition of two-body correction",
// the factor that multiplies rho in V), split into fp16 (2 parts) or bf16 (3 parts) and stored
// K-major as the A operand of the step (b) GEMM, row x * gcp + il (il = i - i0):
//     fp16: G[row][j / 64][part][j % 64]  (128-byte runs of 64 points of one part, 128-byte swizzle
//           tiles, so that one TMA row request moves 128 bytes);
//     bf16: G[part][row][j]               (one plane per part, 64-byte swizzle tiles).
// Computing G once per chunk, instead of inside every orbital-pair tile of the GEMM, removes the
// gradient from the GEMM's critical path; the table costs one HBM write and is then read through L2
// by the GEMM's tiles.
//
// One warp owns a unit of 16 outer points (two lanes each, one per half of a block, its per-point coefficients
// in registers) and a run of inner-point blocks of 32.  For each block it evaluates the gradient in FP32 (two
// inner points per packed FP32 instruction for up to two Jastrow centres; reciprocal square roots
// and reciprocals refined by a Newton-Raphson step, so that no one-signed error of the hardware
// approximations enters the gradient), splits
// it, writes the tiles of the three components (16 rows x 128 bytes, or 3 parts x 16 rows x 64
// bytes) into shared memory in their swizzle (conflict-free 16-byte stores) and one lane stores
// them with TMA.  The fp16 split is exact on a per-range quantum (simt_pack.cuh): for every row and
// accumulation range of the GEMM (RB blocks of 32 inner points), hi = an integer of at most 9
// bits times the range's quantum, lo = the fp16 remainder.  The lanes first stage the FP32 values of
// two blocks (64 points, a hi and a lo tile per component; four blocks when RB = 4) in their tile rows,
// then split them with the quantum of their range's maximum.
//
// What bounds it: the latency of the table loads and of the dependent FP32 chain, so warps in flight count, and
// the staging limits those: with 32 rows a warp (24 KB) an SM held 8 warps and issued in 28 % of its cycles,
// with 16 rows (12 KB) it holds 16.  The FP64 arithmetic of the coefficients (about 250 operations a
// nucleus on a pipe of two per clock, a third of a unit's time) runs once per outer point, in gcoef_kernel, not once per
// unit.  Measured (one GB300), before -> now: 4,000 x 4,000 points and 3 nuclei 253 -> 119 us (with units of 16 blocks, see
// launch_rb), 20,000 x 20,000 and 3 nuclei 3.35 -> 1.75 ms, the bf16 parts of 40,000 x 40,000 points 14.0 -> 9.0 ms.
// The gradient is taken with the pair formula of jastrow_coef.cuh: per-point coefficients times
// polynomials in b = r12 / (1 + r12) and a_jI = |r_j - R_I| / (1 + |r_j - R_I|).
#include <algorithm>

#include "jastrow_coef.cuh"
#include "ptx_sm100.cuh"
#include "simt_pack.cuh"
#include "xtc_internal.cuh"

namespace xtc {
namespace {

constexpr int GF_ROWS = GFIELD_ROWS;       // outer points of a warp
constexpr int GF_WARPS = 4;                // warps of a CTA
constexpr int GF_TILE = GF_ROWS * 64;      // one part's share of a component tile: 16 rows of 64 bytes
// fp16: bits of the integer hi part of G on its range's quantum (|k| <= 2^9, exact in fp16)
constexpr int GF_EXACT_BITS = GEMM_BITS_A;

__device__ __forceinline__ void tma_store_3d(const CUtensorMap* tm, uint32_t src, int c0, int c1, int c2) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(tm)),
               "r"(src), "r"(c0), "r"(c1), "r"(c2)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Waits until the shared memory of every committed bulk store has been read.
__device__ __forceinline__ void bulk_wait_read_all() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
// Waits until every committed bulk store has completed.
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// Nuclei of the kernel's template for n nuclei, and CTAs of an SM (registers: 128 up to 3 nuclei).
constexpr int nuc_slots(int n) { return n <= 4 ? n : 8; }
constexpr int gf_ctas(int nnuc) { return nnuc <= 3 ? 4 : (nnuc == 4 ? 3 : 2); }

// Coefficients of the outer points [i0, i0 + rows), rows past the chunk's n_i repeating its last point:
// coef[k][row], k = 0..13 the point's, 14..16 the low parts of its coordinates (the pair difference is taken
// in hi/lo FP32), then NUC_COEF per nucleus.
template <int NNUC>
__global__ void __launch_bounds__(128) gcoef_kernel(const GfieldArgs args) {
  const int64_t il = blockIdx.x * 128ll + threadIdx.x;
  if (il >= args.rows) return;
  const int64_t ig = args.i0 + (il < args.n_i ? il : args.n_i - 1);
  float pc[PT_COEF];
  float nc[NNUC * NUC_COEF];
  const double gx = args.grid[3 * ig], gy = args.grid[3 * ig + 1], gz = args.grid[3 * ig + 2];
  point_coefs_fixed<float, NNUC>(*args.jp, gx, gy, gz, static_cast<double>(args.g_scale), pc, nc);
  float* o = args.coef + il;
#pragma unroll
  for (int k = 0; k < PT_COEF; ++k) o[k * args.rows] = pc[k];
  o[(PT_COEF + 0) * args.rows] = static_cast<float>(gx - static_cast<double>(pc[0]));
  o[(PT_COEF + 1) * args.rows] = static_cast<float>(gy - static_cast<double>(pc[1]));
  o[(PT_COEF + 2) * args.rows] = static_cast<float>(gz - static_cast<double>(pc[2]));
#pragma unroll
  for (int k = 0; k < NNUC * NUC_COEF; ++k) o[(PT_COEF + 3 + k) * args.rows] = nc[k];
}

template <int PARTS, int NNUC, int RB>
__global__ void __launch_bounds__(GF_WARPS * 32, gf_ctas(NNUC))
    gfield_kernel(const __grid_constant__ CUtensorMap tm_g, const GfieldArgs args) {
  constexpr bool BF16 = PARTS == 3;
  constexpr int JS = NNUC <= 4 ? 12 : 16;  // floats per inner point in the table (launch_jtab)
  constexpr int BLOCK_BYTES = 3 * PARTS * GF_TILE;  // the three component tiles of one block
  constexpr int BB = PARTS == 2 && RB < 2 ? 2 : RB;   // blocks staged together: whole pairs for the fp16 tiles
  constexpr int WARP_BYTES = BB * BLOCK_BYTES;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int row = lane & (GF_ROWS - 1), half = lane / GF_ROWS;  // this lane: points 16 half .. 16 half + 15 of each block
  const int64_t unit = static_cast<int64_t>(blockIdx.x) * GF_WARPS + warp;
  if (unit >= static_cast<int64_t>(args.rows / GF_ROWS) * args.n_seg) return;  // whole warp; no block barrier below
  const int tile = static_cast<int>(unit / args.n_seg), seg = static_cast<int>(unit % args.n_seg);
  const int kb0 = seg * args.kb_per_seg, kb1 = min(args.n_kb, kb0 + args.kb_per_seg);
  const uint32_t buf = smem_u32(smem) + warp * WARP_BYTES;

  const int row0 = tile * GF_ROWS;
  float pc[PT_COEF];
  float nc[NNUC * NUC_COEF];
  const float* cf0 = args.coef + row0 + row;
#pragma unroll
  for (int k = 0; k < PT_COEF; ++k) pc[k] = __ldg(cf0 + k * args.rows);
  const float xl = __ldg(cf0 + (PT_COEF + 0) * args.rows), yl = __ldg(cf0 + (PT_COEF + 1) * args.rows),
              zl = __ldg(cf0 + (PT_COEF + 2) * args.rows);
#pragma unroll
  for (int k = 0; k < NNUC * NUC_COEF; ++k) nc[k] = __ldg(cf0 + (PT_COEF + 3 + k) * args.rows);
  // the same constants duplicated in both halves of a packed pair (paired FP32 path, <= 2 nuclei)
  f32x2 PC[NNUC <= 2 ? PT_COEF : 1], NC[NNUC <= 2 ? NNUC * NUC_COEF : 1], XL = 0, YL = 0, ZL = 0;
  if constexpr (NNUC <= 2) {
#pragma unroll
    for (int k = 0; k < PT_COEF; ++k) PC[k] = pk2(pc[k], pc[k]);
#pragma unroll
    for (int k = 0; k < NNUC * NUC_COEF; ++k) NC[k] = pk2(nc[k], nc[k]);
    XL = pk2(xl, xl);
    YL = pk2(yl, yl);
    ZL = pk2(zl, zl);
  }
  constexpr int NQ = PARTS == 2 ? BB / RB : 1;   // exact ranges staged together
  float gmax[NQ][3];                   // fp16: largest |G| of each range per component
#pragma unroll
  for (int v = 0; v < NQ; ++v) gmax[v][0] = gmax[v][1] = gmax[v][2] = 0.0f;

  for (int kr = kb0; kr < kb1; kr += BB) {
#pragma unroll 1
  for (int rb = 0; rb < BB; ++rb) {
    const int kb = kr + rb;
    // bf16: the block's own tiles; fp16: the hi and lo tiles of the block's pair
    const uint32_t bbuf = buf + (PARTS == 2 ? (rb >> 1) * 2 : rb) * BLOCK_BYTES;
    // 16 records of two inner points each (the pair-interleaved table written by launch_jtab)
    const float* blk = args.jtab + static_cast<int64_t>(kb) * VF_BK * JS;
#pragma unroll 1
    for (int c2 = 0; c2 < 2; ++c2) {
      const int c = 2 * half + c2;   // points 8c .. 8c + 7 of the block
      float gv[3][8];
#pragma unroll
      for (int v2 = 0; v2 < 4; ++v2) {
        const float* rec = blk + (c * 4 + v2) * 2 * JS;  // inner points 8c + 2 v2 and + 1
        if constexpr (NNUC <= 2) {
          f32x2 xh, yh, zh, xlo, ylo, zlo, a0, a1;
          ldg_2x64(rec, xh, yh);
          ldg_2x64(rec + 4, zh, xlo);
          ldg_2x64(rec + 8, ylo, zlo);
          ldg_2x64(rec + 12, a0, a1);
          const f32x2 dx = add2(sub2(PC[0], xh), sub2(XL, xlo));
          const f32x2 dy = add2(sub2(PC[1], yh), sub2(YL, ylo));
          const f32x2 dz = add2(sub2(PC[2], zh), sub2(ZL, zlo));
          const f32x2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
          float r2a, r2b;
          up2(r2, r2a, r2b);
          // unit vector of r1 - r2 taken as zero below 1e-14 bohr (coincident points)
          f32x2 rinv = rsqrt_nr2(fmaxf(r2a, 1e-28f), fmaxf(r2b, 1e-28f));
          {
            float ia, ib;
            up2(rinv, ia, ib);
            rinv = pk2(r2a > 1e-28f ? ia : 0.0f, r2b > 1e-28f ? ib : 0.0f);
          }
          const f32x2 rr = mul2(r2, rinv);
          float ra, rb;
          up2(rr, ra, rb);
          const f32x2 q = rcp_nr2(1.0f + ra, 1.0f + rb);
          const f32x2 b = mul2(rr, q);
          const f32x2 sfac = mul2(mul2(q, q), rinv);
          f32x2 ex = fma2(b, fma2(b, PC[9], PC[6]), PC[3]);
          f32x2 ey = fma2(b, fma2(b, PC[10], PC[7]), PC[4]);
          f32x2 ez = fma2(b, fma2(b, PC[11], PC[8]), PC[5]);
          f32x2 h1 = PC[12], h2 = PC[13];
#pragma unroll
          for (int I = 0; I < NNUC; ++I) {
            const f32x2* cf = NC + I * NUC_COEF;
            const f32x2 a = I == 0 ? a0 : a1;
            const f32x2 t = fma2(b, fma2(b, fma2(a, cf[8], cf[7]), fma2(a, cf[6], cf[5])), fma2(a, cf[4], cf[3]));
            const f32x2 at = mul2(a, t);
            ex = fma2(at, cf[0], ex);
            ey = fma2(at, cf[1], ey);
            ez = fma2(at, cf[2], ez);
            h1 = fma2(a, fma2(a, cf[10], cf[9]), h1);
            h2 = fma2(a, fma2(a, cf[12], cf[11]), h2);
          }
          const f32x2 hs = mul2(fma2(b, h2, h1), sfac);
          up2(fma2(hs, dx, ex), gv[0][2 * v2], gv[0][2 * v2 + 1]);
          up2(fma2(hs, dy, ey), gv[1][2 * v2], gv[1][2 * v2 + 1]);
          up2(fma2(hs, dz, ez), gv[2][2 * v2], gv[2][2 * v2 + 1]);
        } else {
          const float4 q0 = ldg_f4(rec), q1 = ldg_f4(rec + 4), q2 = ldg_f4(rec + 8);
          float2 ap[NNUC];  // a_jI of both points
#pragma unroll
          for (int I = 0; I < NNUC; ++I) ap[I] = __ldg(reinterpret_cast<const float2*>(rec + 12 + 2 * I));
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float xh = h ? q0.y : q0.x, yh = h ? q0.w : q0.z, zh = h ? q1.y : q1.x;
            const float xlo = h ? q1.w : q1.z, ylo = h ? q2.y : q2.x, zlo = h ? q2.w : q2.z;
            const float dx = (pc[0] - xh) + (xl - xlo);
            const float dy = (pc[1] - yh) + (yl - ylo);
            const float dz = (pc[2] - zh) + (zl - zlo);
            const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            const float rinv = r2 > 1e-28f ? rsqrt_nr(r2) : 0.0f;
            const float rr = r2 * rinv;
            const float q = rcp_nr(1.0f + rr);
            const float b = rr * q;
            const float sfac = q * q * rinv;
            float ex = fmaf(b, fmaf(b, pc[9], pc[6]), pc[3]);
            float ey = fmaf(b, fmaf(b, pc[10], pc[7]), pc[4]);
            float ez = fmaf(b, fmaf(b, pc[11], pc[8]), pc[5]);
            float h1 = pc[12], h2 = pc[13];
#pragma unroll
            for (int I = 0; I < NNUC; ++I) {
              const float* cf = nc + I * NUC_COEF;
              const float a = h ? ap[I].y : ap[I].x;
              const float t = fmaf(b, fmaf(b, fmaf(a, cf[8], cf[7]), fmaf(a, cf[6], cf[5])), fmaf(a, cf[4], cf[3]));
              const float at = a * t;
              ex = fmaf(at, cf[0], ex);
              ey = fmaf(at, cf[1], ey);
              ez = fmaf(at, cf[2], ez);
              h1 = fmaf(a, fmaf(a, cf[10], cf[9]), h1);
              h2 = fmaf(a, fmaf(a, cf[12], cf[11]), h2);
            }
            const float hs = fmaf(b, h2, h1) * sfac;
            gv[0][2 * v2 + h] = fmaf(hs, dx, ex);
            gv[1][2 * v2 + h] = fmaf(hs, dy, ey);
            gv[2][2 * v2 + h] = fmaf(hs, dz, ez);
          }
        }
      }
      // the previous range's tiles must have been read by their TMA stores before they are overwritten
      if (c2 == 0 && rb == 0 && kr > kb0) {
        if (lane == 0) bulk_wait_read_all();
        __syncwarp();
      }
      if constexpr (PARTS == 2) {
        // FP32 staging in the row's 128-byte rows of the pair's component tiles: points 8c .. 8c + 7 in
        // the hi tile for even c, the lo tile for odd c, 16-byte chunks b and b + 1 with b = 4 (rb % 2) +
        // 2 half, so that the split below rewrites, for the lane's half of the block, exactly the chunks
        // that the lane itself has written and read; and the range maxima
        const int b = (rb & 1) * 4 + half * 2;
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          float m = 0.0f;
#pragma unroll
          for (int k = 0; k < 8; ++k) m = fmaxf(m, fabsf(gv[x][k]));
#pragma unroll
          for (int v = 0; v < NQ; ++v)
            if (NQ == 1 || rb == v) gmax[v][x] = fmaxf(gmax[v][x], m);
          const uint32_t trow = bbuf + (2 * x + c2) * 2 * GF_TILE;
          st_shared_v4(trow + sw128_offset(row, b), __float_as_uint(gv[x][0]), __float_as_uint(gv[x][1]),
                       __float_as_uint(gv[x][2]), __float_as_uint(gv[x][3]));
          st_shared_v4(trow + sw128_offset(row, b + 1), __float_as_uint(gv[x][4]), __float_as_uint(gv[x][5]),
                       __float_as_uint(gv[x][6]), __float_as_uint(gv[x][7]));
        }
      } else {
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          uint32_t w[4][PARTS];
#pragma unroll
          for (int h = 0; h < 4; ++h) split_pair<BF16>(gv[x][2 * h], gv[x][2 * h + 1], w[h]);
#pragma unroll
          for (int p = 0; p < PARTS; ++p)
            st_shared_v4(bbuf + (x * PARTS + p) * GF_TILE + sw64_offset(row, c), w[0][p], w[1][p], w[2][p], w[3][p]);
        }
      }
    }
  }
    if constexpr (PARTS == 2) {
      // exact split of the lane's values per component on their range's quantum (the maximum over both of the
      // row's lanes): hi of points 8c .. 8c + 7 of the pair's block rb goes to chunk 4 (rb % 2) + c of the hi tile, lo to the
      // same chunk of the lo tile (tiles of 16 rows x 128 bytes, the layout the GEMM loads)
#pragma unroll
      for (int x = 0; x < 3; ++x) {
#pragma unroll
        for (int rb = 0; rb < BB; ++rb) {
          if (NQ > 1 || rb == 0) {
            float& m = gmax[NQ == 1 ? 0 : rb][x];
            m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, GF_ROWS));
          }
          const int q = exact_quantum(gmax[NQ == 1 ? 0 : rb][x], GF_EXACT_BITS);
          const uint32_t hi = buf + (rb >> 1) * 2 * BLOCK_BYTES + 2 * x * 2 * GF_TILE, lo = hi + 2 * GF_TILE;
          const uint32_t c0 = sw128_offset(row, 4 * (rb & 1) + 2 * half), c1 = sw128_offset(row, 4 * (rb & 1) + 2 * half + 1);
          uint32_t f[16];
          ld_shared_v4(hi + c0, f[0], f[1], f[2], f[3]);
          ld_shared_v4(hi + c1, f[4], f[5], f[6], f[7]);
          ld_shared_v4(lo + c0, f[8], f[9], f[10], f[11]);
          ld_shared_v4(lo + c1, f[12], f[13], f[14], f[15]);
          uint32_t w[8][2];
#pragma unroll
          for (int k = 0; k < 8; ++k)
            split_pair_exact(__uint_as_float(f[2 * k]), __uint_as_float(f[2 * k + 1]), q, w[k]);
          st_shared_v4(hi + c0, w[0][0], w[1][0], w[2][0], w[3][0]);
          st_shared_v4(hi + c1, w[4][0], w[5][0], w[6][0], w[7][0]);
          st_shared_v4(lo + c0, w[0][1], w[1][1], w[2][1], w[3][1]);
          st_shared_v4(lo + c1, w[4][1], w[5][1], w[6][1], w[7][1]);
        }
      }
#pragma unroll
      for (int v = 0; v < NQ; ++v) gmax[v][0] = gmax[v][1] = gmax[v][2] = 0.0f;
    }
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) {
      if constexpr (PARTS == 2) {
#pragma unroll
        for (int pr = 0; pr < BB / 2; ++pr)
#pragma unroll
          for (int t = 0; t < 6; ++t)  // component t / 2, part t % 2
            tma_store_3d(&tm_g, buf + (2 * pr) * BLOCK_BYTES + t * 2 * GF_TILE, (kr / 2 + pr) * 128 + (t & 1) * 64,
                         static_cast<int>((t >> 1) * args.gcp) + row0, 0);
      } else {
#pragma unroll
        for (int rb = 0; rb < BB; ++rb)
#pragma unroll
          for (int t = 0; t < 3 * PARTS; ++t)  // component t / PARTS, part t % PARTS
            tma_store_3d(&tm_g, buf + rb * BLOCK_BYTES + t * GF_TILE, (kr + rb) * VF_BK,
                         static_cast<int>((t / PARTS) * args.gcp) + row0, t % PARTS);
      }
      bulk_commit();
    }
  }
  if (lane == 0) bulk_wait_all();
  __syncwarp();
}

template <int PARTS, int NNUC, int RB>
void launch_rb(const CUtensorMap* tm, const GfieldArgs& in, cudaStream_t st) {
  auto kern = gfield_kernel<PARTS, NNUC, RB>;
  constexpr int bb = PARTS == 2 && RB < 2 ? 2 : RB;
  constexpr int smem = GF_WARPS * bb * 3 * PARTS * GF_TILE + 1024;  // warps x staged blocks of three tiles
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  GfieldArgs a = in;
  // Blocks per unit (a multiple of 4: whole staged groups): the length with the least (rounds of resident warps) x
  // (blocks + 1 for the coefficients), the longest of equals.  124 blocks of 248 tiles: 16 (one round), not 32.
  const int64_t tiles = a.rows / GF_ROWS, slots = static_cast<int64_t>(std::max(a.n_sm, 1)) * gf_ctas(NNUC) * GF_WARPS;
  int64_t best_cost = -1;
  for (int seg = 4; seg <= 64; seg += 4) {
    const int64_t units = tiles * ((a.n_kb + seg - 1) / seg), cost = (units + slots - 1) / slots * (seg + 1);
    if (best_cost < 0 || cost <= best_cost) {
      best_cost = cost;
      a.kb_per_seg = seg;
    }
  }
  a.n_seg = (a.n_kb + a.kb_per_seg - 1) / a.kb_per_seg;
  const int64_t units = tiles * a.n_seg;
  const unsigned blocks = static_cast<unsigned>((units + GF_WARPS - 1) / GF_WARPS);
  gcoef_kernel<NNUC><<<static_cast<unsigned>((a.rows + 127) / 128), 128, 0, st>>>(a);
  kern<<<blocks, GF_WARPS * 32, smem, st>>>(*tm, a);
}
template <int PARTS, int NNUC>
void launch_t(const CUtensorMap* tm, const GfieldArgs& a, cudaStream_t st) {
  if (PARTS == 2 && a.range_blocks == 4)
    launch_rb<PARTS, NNUC, 4>(tm, a, st);
  else if (PARTS == 2 && a.range_blocks == 2)
    launch_rb<PARTS, NNUC, 2>(tm, a, st);
  else
    launch_rb<PARTS, NNUC, 1>(tm, a, st);
}

}  // namespace

size_t gfield_coef_floats(int n_nuc, int64_t rows) {
  return static_cast<size_t>(PT_COEF + 3 + nuc_slots(n_nuc) * NUC_COEF) * rows;
}

void launch_gfield(const CUtensorMap* tm_g_store, const GfieldArgs& a, int parts, cudaStream_t st) {
  if (a.rows <= 0 || a.n_kb <= 0) return;
  if (parts == 2) {
    switch (a.n_nuc) {
      case 1: launch_t<2, 1>(tm_g_store, a, st); break;
      case 2: launch_t<2, 2>(tm_g_store, a, st); break;
      case 3: launch_t<2, 3>(tm_g_store, a, st); break;
      case 4: launch_t<2, 4>(tm_g_store, a, st); break;
      default: launch_t<2, 8>(tm_g_store, a, st); break;  // 5..8 nuclei
    }
  } else {
    switch (a.n_nuc) {
      case 1: launch_t<3, 1>(tm_g_store, a, st); break;
      case 2: launch_t<3, 2>(tm_g_store, a, st); break;
      case 3: launch_t<3, 3>(tm_g_store, a, st); break;
      case 4: launch_t<3, 4>(tm_g_store, a, st); break;
      default: launch_t<3, 8>(tm_g_store, a, st); break;  // 5..8 nuclei
    }
  }
}

}  // namespace xtc
