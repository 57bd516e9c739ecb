// Step (b) on the tensor cores: the vector pair fields of the "Decomposition of two-body
// correction" section,
//     V_x[i][pq] = sum_j G_x(i, j) rho^T[pq][j],   G_x(i, j) = d/dx_i u(r_i, r_j),
//     rho^T[pq][j] = w_j phi_p(j) phi_q(j),
// as a split-precision GEMM over the inner points j: A = G (written by gfield.cu, rows x*gcp + il),
// B = rho^T (written by the rho split kernel), K-major, all operands loaded by TMA.  The same fp16
// engine runs step (d) of Appendix B (MODE 1): M += L^T R with A = the split rows L[pq]
// (rho, V) and B = the split rows R[rs] (A, B) of a chunk, K = 4 x chunk points, each row carrying
// its own power-of-2 scale; its tile sums are added into M[pq][rs] by assemble_finalize_kernel.
//
// fp16 x2 engine (xgemm_kernel).  Both operands are split exactly on per-range quanta (simt_pack.cuh):
// per row and accumulation range of kd stages (kd * 32 K values), hi = an integer times the row's
// power-of-2 quantum for that range (from the range's largest magnitude), lo = the fp16 remainder,
// with bit widths such that the range's hi x hi products sum within 2^24 units.
// The tensor core's FP32 accumulator truncates toward zero at every MMA, which biases a long sum
// by a relative ~2^-24 per MMA, always toward zero; the hi x hi sums of a range are exact, so they
// go, one range at a time, into an accumulator E, which the drain warps add into FP32 running sums
// (round to nearest) after every range.  The cross products (about 2^-9 of the total, signs that
// follow the rounding remainders rather than the data) go into a second accumulator X, drained
// every `xper` stages; their truncation is 2^-9 smaller and does not accumulate one-sided.  They
// must include lo_a x lo_b: where both operands hold values far below their range's maximum, hi is
// 0 and lo is the whole value.  Both steps issue hi_a x lo_b and lo_a x fp16(b), with fp16(b) a
// third plane of the B operand (rho^T in step (b), R in step (d)): lo_a x (hi_b + lo_b) to within
// fp16's rounding of b (a relative 2^-12 of a term that is itself 2^-10 of the product), one
// product where two would be needed.
//
// Tile 128 A rows x 128 columns, 32 K values per stage, both parts of a row of a block in one
// 128-byte row of 64 values per part: [row][K / 64][hi, lo][64].
//
// Tile and split of the work.  With one CTA per 128 x 128 tile the engine was bound by shared
// memory: per 32 values of K the six MMAs read 48 KB of operands and the loads wrote 40 KB, 704 cycles
// at 128 bytes per clock (705 measured) for 384 cycles of tensor pipe.  Two things cut that: pairs of
// CTAs share a 256 x 128 tile (tcgen05 cta_group::2: 256 rows of A, each CTA loads half of B), and
// hi_a x hi_b and hi_a x lo_b are one MMA of 256 columns, [hi_b | lo_b], with hi_b in the leader's shared
// memory and lo_b in the other's, writing the adjacent accumulators [E | X], so hi_a is read once.  Per
// 64 values and CTA: 56 KB read, 56 KB written, 875 cycles for 768 of tensor pipe.
//   * warp 0 of each CTA (one lane): TMA loads (4 stages of 56 KB: hi and lo of A, one part of B, half of
//     fp16(B)), completing on the leader's barriers; a slot is reloaded once its MMAs have completed;
//   * warps 1 and 2 of the leader: the MMAs of the even / odd ranges into the accumulator sets (E0, X0) and
//     (E1, X1) (4 x 128 of 512 TMEM columns in each CTA), so that one set is drained while
//     the other fills; commits (to both CTAs) after every stage and every range;
//   * warps 3..18 of each CTA: after every range, drains of E_k, and every `xper` blocks of X_k, into FP32
//     running sums held in registers (four warps per TMEM lane quarter, 32 columns each); what was
//     read is set to zero, so that every MMA accumulates.  The
//     sums move into an FP64 accumulator in HBM, private to the CTA and column-major in its tile,
//     one column per range in turn (each column at least once per `flush` ranges; each element
//     belongs to one thread); vfield_finalize_kernel writes V from it (MODE 0).
// Tiles are ordered in groups of GM row tiles so that the CTAs resident at one time share their A
// and B panels in L2.
//
// bf16 x3 engine (vfield_bf16_kernel, step (b) of the bf16 precision): three bf16 planes per
// operand (64-byte swizzle), six products (i + j <= 2) into one of two TMEM accumulators per range
// of `kd` stages, small cross products first, drained into FP32 running sums after every range.
// Its accumulation is not exact: the truncation bias is only kept small by the short ranges.
#include <algorithm>

#include "gemm_rules.h"
#include "ptx_sm100.cuh"
#include "xtc_internal.cuh"

namespace xtc {
namespace {

constexpr int DRAIN_WARPS = 8;       // two per TMEM lane quarter, half of the columns each
constexpr int GM = 16;               // row tiles per group (L2 reuse of the column panels)
constexpr int NRB = 8;               // per-stage / per-range barriers (stage or range r uses r % NRB)

__device__ __forceinline__ void red_add_f64(double* p, double v) {
  asm volatile("red.global.add.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}

// 32 lanes x 16 consecutive 32-bit columns: thread t of the warp receives lane (base + t).
__device__ __forceinline__ void tmem_ld_x16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}

// Tile coordinates of CTA L in the grouped order (GM row tiles x every column tile, row fastest).
struct TileXY {
  int m_tile, n_tile;
};
template <int G = GM>
__device__ __forceinline__ TileXY grouped_tile(int L, int m_tiles, int n_tiles) {
  const int group = L / (G * n_tiles);
  const int first_m = group * G;
  const int gm = min(G, m_tiles - first_m);
  const int rem = L - group * G * n_tiles;
  return {first_m + rem % gm, rem / gm};
}

// Tile of CTA L of the fp16 engine: consecutive CTAs are the two row tiles of a pair; groups of GM row
// tiles x every column tile, pair row fastest.  With an odd number of row tiles the last pair's second
// tile does not exist (m_tile == m_tiles).
__device__ __forceinline__ TileXY pair_tile(int L, int m_tiles, int n_tiles) {
  const TileXY t = grouped_tile<GM / 2>(L >> 1, (m_tiles + 1) >> 1, n_tiles);
  return {2 * t.m_tile + (L & 1), t.n_tile};
}

// =================================================================== fp16 x2 engine
constexpr int XB_BN = 128;                        // tile columns
constexpr int XB_BK = 64;                         // K values per stage
constexpr int XB_DRAIN_WARPS = 16;                // four per TMEM lane quarter, a quarter of the columns each
constexpr int XB_HC = XB_BN / 4;                  // running-sum columns per drain thread
constexpr int XB_PART = VF_BM * XB_BK * 2;        // 128 rows of 128 bytes: hi or lo of A, hi (leader) or lo of B
constexpr int XB_B16_BYTES = XB_BN / 2 * XB_BK * 2;  // fp16(B), half of the columns in each CTA
constexpr int XB_STAGE = 3 * XB_PART + XB_B16_BYTES;
constexpr int XB_STAGES = 4;
constexpr int XB_THREADS = (3 + XB_DRAIN_WARPS) * 32;  // TMA warp, two MMA warps, drains
constexpr int XB_SMEM = XB_STAGES * XB_STAGE + 1024 + 256;
constexpr int XB_SET = 2 * XB_BN;                 // TMEM columns of an accumulator set (E, X)
static_assert(XB_BN == vf_bn(2), "tile width of the fp16 engine");
static_assert(2 * XB_SET <= 512, "E0, X0, E1, X1 in 512 TMEM columns");
static_assert(XB_HC == 32, "drain columns per thread (one 32-column load)");
static_assert(XB_SMEM <= 232448, "shared memory per CTA");
static_assert((2 * XB_STAGES + 5) * 8 + 8 <= 256, "barrier area");

// Shared-memory descriptor of a K-major operand in the 128-byte swizzle, for a shared address
// below 2^18: the constant fields plus the address in 16-byte units (a plain add per stage and
// K step, no re-encoding in the issue loop).
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) { return sdesc_kmajor_sw128(0) + (saddr >> 4); }

template <int MODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(XB_THREADS, 1)
    xgemm_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                 const __grid_constant__ CUtensorMap tm_b16, const VfieldArgs args) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + XB_STAGES * XB_STAGE);
  uint64_t* full = bars;                 // [XB_STAGES] leader: the stage's loads of both CTAs landed
  uint64_t* sfree = full + XB_STAGES;    // [XB_STAGES] the stage's MMAs completed (slot free)
  uint64_t* rdone = sfree + XB_STAGES;   // [2] every MMA of the range in accumulator set k completed
  uint64_t* e_free = rdone + 2;          // [2] leader: the drains of both CTAs released set k, zeroed
  uint64_t* fin_bar = e_free + 2;        // leader: every MMA completed
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(fin_bar + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // warp: uniform
  const uint32_t rank = cluster_rank();
  const int m_tiles = MODE == 0 ? 3 * args.mt_per_x : (args.rows_a + VF_BM - 1) / VF_BM;
  const TileXY t = pair_tile(args.cta0 + blockIdx.x, m_tiles, args.n_tiles);
  const bool valid = t.m_tile < m_tiles;          // a tile that does not exist repeats the last one's rows
  const int m_tile = valid ? t.m_tile : m_tiles - 1;
  // mode 0: rows x * gcp + outer point of component x; mode 1: rows pq
  const int x = MODE == 0 ? m_tile / args.mt_per_x : 0;
  const int ib = MODE == 0 ? (m_tile - x * args.mt_per_x) * VF_BM : m_tile * VF_BM;
  const int row0 = MODE == 0 ? static_cast<int>(x * args.gcp) + ib : ib;
  const int split = blockIdx.y;
  const int kb0 = split * args.kb_per_split;               // multiple of 2 and of kd
  // MODE 1: slices of the chain, each but the last running XB_HC ranges into the next one (chain_slices)
  const int kb_over = MODE == 1 && args.slices > 1 ? XB_HC * args.kd : 0;
  const int n_it = min(args.n_kb, kb0 + args.kb_per_split + kb_over) - kb0;  // blocks of 32 K values, even
  const int n_st = (n_it + 1) >> 1;                        // stages
  const int kd = args.kd;                                  // blocks per exact range (1, 2 or 4)
  const int n_ranges = (n_it + kd - 1) / kd;
  const int xr = max(1, args.xper / (2 * kd));             // ranges of one set per X drain

  if (threadIdx.x == 0) {
    for (int s = 0; s < XB_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&sfree[s], args.kd == 1 ? 2 : 1);  // commits per stage: one of each issuer when they share it
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(&rdone[k], 1);
      mbar_init(&e_free[k], 2 * XB_DRAIN_WARPS);
    }
    mbar_init(fin_bar, 2);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tm_a);
    tma_prefetch_desc(&tm_b);
    tma_prefetch_desc(&tm_b16);
  }
  if (warp == 0) tmem_alloc_pair(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);

  if (warp == 0) {
    if (lane == 0) {
      // ---------------------------------------------------------------- TMA producer (both CTAs)
      // own 128 rows of A (hi and lo), one part of B's 128 columns (hi in the leader, lo in the other
      // CTA) and half of fp16(B); both CTAs' loads complete on the leader's barrier
      int issued = 0;
      for (int it = 0; it < n_st; ++it) {
        const int s = it % XB_STAGES;
        if (it >= XB_STAGES &&
            !mbar_wait(&sfree[s], ((it / XB_STAGES) - 1) & 1, abort_flag, args.err, DEV_ERR_TIMEOUT_VF))
          break;
        if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * XB_STAGE);
        const uint32_t bar = cluster_addr(&full[s], 0);
        uint8_t* st = smem + s * XB_STAGE;
        const int k0 = kb0 * VF_BK + it * XB_BK;
        tma_load_3d_pair(st, &tm_a, bar, 2 * k0, row0, 0);
        tma_load_3d_pair(st + XB_PART, &tm_a, bar, 2 * k0 + XB_BK, row0, 0);
        tma_load_3d_pair(st + 2 * XB_PART, &tm_b, bar, 2 * k0 + static_cast<int>(rank) * XB_BK, t.n_tile * XB_BN, 0);
        tma_load_3d_pair(st + 3 * XB_PART, &tm_b16, bar, k0, t.n_tile * XB_BN + static_cast<int>(rank) * (XB_BN / 2), 0);
        issued = it + 1;
      }
      // The last slots come free once their MMAs have read them, so every copy has landed and every
      // arrival on this CTA's barriers has been made before the CTA exits.  After an abort the leader waits
      // for the loads it announced instead, and the other CTA (whose loads complete on the leader's
      // barriers) for a time no copy takes.
      int zero = 0;
      volatile int* no_abort = reinterpret_cast<volatile int*>(&zero);
      for (int it = max(0, issued - XB_STAGES); it < issued; ++it)
        if (!mbar_wait(&sfree[it % XB_STAGES], (it / XB_STAGES) & 1, abort_flag, args.err, DEV_ERR_TIMEOUT_VF)) break;
      if (*abort_flag) {
        if (rank == 0) {
          for (int it = max(0, issued - XB_STAGES); it < issued; ++it)
            mbar_wait(&full[it % XB_STAGES], (it / XB_STAGES) & 1, no_abort, args.err, DEV_ERR_TIMEOUT_VF);
        } else {
          const unsigned long long t0 = global_timer_ns();
          while (global_timer_ns() - t0 < 50000000ull) {
          }
        }
      }
    }
  } else if (warp == 1 || warp == 2) {
    if (rank == 0) {
      // ---------------------------------------------------------------- MMA issuers (leader)
      // Issuer k takes the ranges r = k, k + 2, ... into set k (one thread's waits and instructions for a
      // range take about 1,500 cycles, twice its MMAs): per block of 32 values and k-step of 16, hi_a x [hi_b | lo_b] in
      // one 256-column MMA into [E_k | X_k], then lo_a x fp16(b) into X_k (fp16(b): lo_a x (hi_b + lo_b)
      // to within fp16's rounding).  The drains zero E_k after every range and X_k after its period, so
      // that every MMA accumulates.
      constexpr uint32_t idesc_hi = idesc_f16(2 * VF_BM, 2 * XB_BN, false);
      constexpr uint32_t idesc_lo = idesc_f16(2 * VF_BM, XB_BN, false);
      const uint32_t smem_base = smem_u32(smem);
      bool alive = true;
      const int k = warp - 1;
      const uint32_t set = tmem + k * XB_SET;
      const uint32_t sfree_bar = smem_base + XB_STAGES * XB_STAGE + XB_STAGES * 8, rdone_bar = sfree_bar + (XB_STAGES + k) * 8;
      for (int r = k, u = 0; r < n_ranges && alive; r += 2, ++u) {
        const int it0 = r * kd, it1 = min(n_it, it0 + kd);
        const bool x_end = u % xr == xr - 1 || r + 2 >= n_ranges;
        for (int it = it0; it < it1; ++it) {
          const int s = (it >> 1) % XB_STAGES;
          // the stage first: it landed long ago as a rule, the set is what the issuer waits for
          if (!(it & 1) || it == it0)
            alive = mbar_spin_warp(&full[s], ((it >> 1) / XB_STAGES) & 1, abort_flag, args.err, DEV_ERR_TIMEOUT_VF);
          // (a vote at every poll of e_free: 3 % less for N = 120 and small builds, but 4 % more for pieces of N = 200, whose
          // CTAs drift apart faster than their launches line them up)
          if (it == it0) alive = alive && mbar_spin_vote(&e_free[k], u & 1, abort_flag, args.err, DEV_ERR_TIMEOUT_VF);
          if (!alive) break;
          tc_fence_after();
          // the block's 32 values are half of the 128-byte rows; k-steps of 16 values advance 32 bytes
          const uint64_t ah = sw128_desc(smem_base + s * XB_STAGE) + (it & 1) * 4;
          const uint64_t al = ah + (XB_PART >> 4), b = ah + (2 * XB_PART >> 4), b16 = ah + (3 * XB_PART >> 4);
          tc_mma_f16_pair(set, ah, b, idesc_hi);
          tc_mma_f16_pair(set, ah + 2, b + 2, idesc_hi);
          // E_k is complete here: its drain need not wait for the last cross products, unless it takes X_k too
          if (it == it1 - 1 && !x_end) tc_commit_pair(rdone_bar);
          tc_mma_f16_pair(set + XB_BN, al, b16, idesc_lo);
          tc_mma_f16_pair(set + XB_BN, al + 2, b16 + 2, idesc_lo);
          if ((it & 1) || it == it1 - 1) tc_commit_pair(sfree_bar + s * 8);
        }
        if (alive && x_end) tc_commit_pair(rdone_bar);
      }
      // every MMA of both issuers has completed once fin_bar fires
      tc_commit_pair_local(smem_u32(fin_bar));
      int zero = 0;
      mbar_wait(fin_bar, 0, reinterpret_cast<volatile int*>(&zero), args.err, DEV_ERR_TIMEOUT_VF);
    }
  } else {
    // ------------------------------------------------------------------ drains and epilogue
    const int quarter = warp & 3;               // TMEM lanes 32*quarter .. +31 (hardware rule)
    const int group = (warp - 3) >> 2;          // columns XB_HC*group .. +XB_HC-1
    const uint32_t c_base = static_cast<uint32_t>(group * XB_HC);
    const uint32_t my = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + c_base;
    const uint32_t free_bar[2] = {cluster_addr(&e_free[0], 0), cluster_addr(&e_free[1], 0)};
    float S[XB_HC];
#pragma unroll
    for (int k = 0; k < XB_HC; ++k) S[k] = 0.0f;
    // the accumulators start at zero
#pragma unroll
    for (int a = 0; a < 4; ++a) tmem_zero_x32(my + a * XB_BN);
    tmem_wait_st();
    tc_fence_before();
    __syncwarp();
    if (lane == 0) {
      mbar_arrive_cluster(free_bar[0]);
      mbar_arrive_cluster(free_bar[1]);
    }
    // The FP32 running sums move into the CTA-private FP64 accumulator, column-major in the tile:
    // Vacc[(split * gridDim.x + tile) * 128 * BN + column * 128 + row], column = c_base + c.  Column
    // c of every thread goes after range r when r % flush == c (staggered, so that no drain carries a
    // whole tile of FP64 adds at once): a store the first time (r < flush), then a fire-and-forget
    // reduction; every column is flushed at least once per `flush` ranges.
    double* acc = args.Vacc + (static_cast<int64_t>(split) * args.n_cta + args.cta0 + blockIdx.x) * VF_BM * XB_BN +
                  static_cast<int64_t>(c_base) * VF_BM + quarter * 32 + lane;
    auto flush_col = [&](int c, bool first) {
#pragma unroll
      for (int k = 0; k < XB_HC; ++k)
        if (k == c) {
          if (first)
            acc[k * VF_BM] = static_cast<double>(S[k]);
          else
            red_add_f64(acc + k * VF_BM, static_cast<double>(S[k]));
          S[k] = 0.0f;
        }
    };
    // A later slice of the chain starts where column 0 was flushed: column c's sums up to range c belong to the
    // slice before, and its first flush is at range flush + c.
    const int first = MODE == 1 && split > 0 ? args.flush : 0;
    const bool last = MODE == 0 || split + 1 >= args.slices;
    bool ok = true;
    for (int r = 0; r < n_ranges && ok; ++r) {
      const int k = r & 1, u = r >> 1;
      // X_k is drained at the end of each of its periods and after the set's last range
      const bool x_end = u % xr == xr - 1 || r + 2 >= n_ranges;
      // one lane waits, suspended: the board is at its power cap in these kernels, and 16 polling warps cost
      // 10 % of the time (100.7 ms a 9,728-point launch with every lane polling, 95.3 with one, 90.7 so)
      if (lane == 0) ok = mbar_wait(&rdone[k], u & 1, abort_flag, args.err, DEV_ERR_TIMEOUT_VF);
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) break;
      tc_fence_after();
      uint32_t d[32];
      const uint32_t e_col = my + k * XB_SET;
      tmem_ld_32x32b_x32(e_col, d);
      tmem_wait_ld();
      tmem_zero_x32(e_col);
      if (x_end) {
#pragma unroll
        for (int c = 0; c < XB_HC; ++c) S[c] += __uint_as_float(d[c]);
        tmem_ld_32x32b_x32(e_col + XB_BN, d);
        tmem_wait_ld();
        tmem_zero_x32(e_col + XB_BN);
      }
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(free_bar[k]);
      // the sums and the staggered FP64 flush (the accumulators are already handed back to the MMAs)
#pragma unroll
      for (int c = 0; c < XB_HC; ++c) S[c] += __uint_as_float(d[c]);
      if (valid && args.flush > 0 && r % args.flush < XB_HC) {
        if (MODE == 1 && r < first) {
#pragma unroll
          for (int c = 0; c < XB_HC; ++c)
            if (c == r) S[c] = 0.0f;
        } else {
          flush_col(r % args.flush, r < first + args.flush);
        }
      }
    }
    if (MODE == 1 && !last) {
      // what is left belongs to the next slice
    } else if (args.flush > 0) {
      // the remaining sums join the FP64 accumulator (columns never flushed in the loop are
      // stored); a finalize kernel writes V (mode 0) or adds the tile into M (mode 1)
      if (ok && valid) {
#pragma unroll
        for (int c = 0; c < XB_HC; ++c) {
          if (c < min(n_ranges - first, args.flush))
            red_add_f64(acc + c * VF_BM, static_cast<double>(S[c]));
          else
            acc[c * VF_BM] = static_cast<double>(S[c]);
        }
      }
    } else if (MODE == 0) {
      // FP32 sums straight to V: row = outer point ib + row of component x, both (p, s) and (s, p)
      const int row = quarter * 32 + lane;
      const int64_t il = static_cast<int64_t>(ib) + row;
      const int pq0 = t.n_tile * XB_BN + static_cast<int>(c_base);
      if (ok && valid && !*abort_flag && il < args.n_i && n_it > 0) {
        float* Vz = args.V + split * v_slice(args.gcp, args.n_orb);
#pragma unroll
        for (int k = 0; k < XB_HC; ++k) {
          const int pq = pq0 + k;
          if (pq < args.n_pair) {
            const int p = __ldg(args.pair_p + pq), q = __ldg(args.pair_q + pq);
            const float v = ldexpf(S[k] * args.unscale_g, -__ldg(args.colexp + pq));
            Vz[v_index(il, p, q, x, args.n_orb)] = v;
            Vz[v_index(il, q, p, x, args.n_orb)] = v;
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync();  // the pair's MMAs, loads and remote arrivals are done
  if (warp == 0) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc_pair(tmem, 512);
  }
}

// =================================================================== bf16 x3 engine (step (b))
// CTA pairs share a 256 x 160 tile (tcgen05 cta_group::2): each CTA loads its 128 rows of A and 80 of B's
// columns.  One CTA per 128 x 160 tile was bound by shared memory: per 64 values of K the 24 MMAs read 216 KB and the
// loads wrote 108 KB, 2,531 cycles at 128 bytes a clock (3,360 measured) for 1,920 of tensor pipe; a pair's
// CTA reads 156 KB and writes 78 KB, 1,828 (2,410 measured).  Step (b) of a water-sized build (40,000 points, 58
// orbitals, one GB300): 71.6 -> 51.4 ms.
constexpr int BF_BN = 160;
constexpr int BF_HC = BF_BN / 2;
constexpr int BF_PARTS = 3;
constexpr int BF_A_TILE = VF_BM * 64;             // bytes per part of an A tile (128 rows of 64 B)
constexpr int BF_B_TILE = BF_BN / 2 * 64;         // bytes per part of a CTA's half of the B tile
constexpr int BF_STAGE = BF_PARTS * (BF_A_TILE + BF_B_TILE);
constexpr int BF_STAGES = 5;
constexpr int BF_THREADS = (2 + DRAIN_WARPS) * 32;
constexpr int BF_SMEM = BF_STAGES * BF_STAGE + 1024 + 256;
static_assert(BF_BN == vf_bn(3), "tile width of the bf16 engine");
static_assert(BF_STAGE % 1024 == 0 && BF_B_TILE % 512 == 0, "swizzle atoms");
static_assert(BF_SMEM <= 232448, "shared memory per CTA");
static_assert(NRB > BF_STAGES, "range barriers");
static_assert(2 * BF_BN <= 512 && BF_BN % 32 == 0, "two accumulators, drain halves of 16-column chunks");

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(BF_THREADS, 1)
    vfield_bf16_kernel(const __grid_constant__ CUtensorMap tm_g, const __grid_constant__ CUtensorMap tm_rho,
                       const VfieldArgs args) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + BF_STAGES * BF_STAGE);
  uint64_t* full = bars;                      // [BF_STAGES] leader: the stage's loads of both CTAs landed
  uint64_t* rdone = full + BF_STAGES;         // [NRB] the MMAs of range r (r % NRB) completed
  uint64_t* d_free = rdone + NRB;             // [2] leader: the drains of both CTAs released accumulator b
  uint64_t* fin_bar = d_free + 2;             // leader: every MMA completed
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(fin_bar + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // warp: uniform
  const uint32_t rank = cluster_rank();
  const int m_tiles = 3 * args.mt_per_x;
  const TileXY t = pair_tile(args.cta0 + blockIdx.x, m_tiles, args.n_tiles);
  const bool valid = t.m_tile < m_tiles;          // a tile that does not exist repeats the last one's rows
  const int m_tile = valid ? t.m_tile : m_tiles - 1;
  const int x = m_tile / args.mt_per_x;
  const int ib = (m_tile - x * args.mt_per_x) * VF_BM;
  const int row0 = static_cast<int>(x * args.gcp) + ib;
  const int split = blockIdx.y;
  const int kb0 = split * args.kb_per_split;
  const int n_it = min(args.n_kb, kb0 + args.kb_per_split) - kb0;
  const int kd = args.kd;
  const int n_ranges = (n_it + kd - 1) / kd;

  if (threadIdx.x == 0) {
    for (int s = 0; s < BF_STAGES; ++s) mbar_init(&full[s], 1);
    for (int r = 0; r < NRB; ++r) mbar_init(&rdone[r], 1);
    for (int b = 0; b < 2; ++b) mbar_init(&d_free[b], 2 * DRAIN_WARPS);
    mbar_init(fin_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tm_g);
    tma_prefetch_desc(&tm_rho);
  }
  if (warp == 0) tmem_alloc_pair(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);
  const uint32_t smem_base = smem_u32(smem);

  if (warp == 0) {
    if (lane == 0) {
      // ---------------------------------------------------------------- TMA producer (both CTAs)
      int seen = 0;  // ranges known to have completed (their slots are free again)
      bool ok = true;
      const int n0 = t.n_tile * BF_BN + static_cast<int>(rank) * (BF_BN / 2);
      for (int it = 0; it < n_it && ok; ++it) {
        const int s = it % BF_STAGES;
        if (it >= BF_STAGES) {
          const int need = (it - BF_STAGES) / kd;  // range holding the slot's previous stage
          for (; seen <= need && ok; ++seen)
            ok = mbar_wait(&rdone[seen % NRB], (seen / NRB) & 1, abort_flag, args.err, DEV_ERR_TIMEOUT_VF);
          if (!ok) break;
        }
        if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * BF_STAGE);
        const uint32_t bar = cluster_addr(&full[s], 0);
        uint8_t* st = smem + s * BF_STAGE;
        for (int p = 0; p < BF_PARTS; ++p) {
          tma_load_3d_pair(st + p * BF_A_TILE, &tm_g, bar, (kb0 + it) * VF_BK, row0, p);
          tma_load_3d_pair(st + BF_PARTS * BF_A_TILE + p * BF_B_TILE, &tm_rho, bar, (kb0 + it) * VF_BK, n0, p);
        }
      }
      // Every range completes before the CTA exits, so every copy has landed and every arrival on this CTA's
      // barriers has been made.  After an abort: a time no copy takes.
      for (; ok && seen < n_ranges; ++seen)
        ok = mbar_wait(&rdone[seen % NRB], (seen / NRB) & 1, abort_flag, args.err, DEV_ERR_TIMEOUT_VF);
      if (!ok || *abort_flag) {
        const unsigned long long t0 = global_timer_ns();
        while (global_timer_ns() - t0 < 50000000ull) {
        }
      }
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // ---------------------------------------------------------------- MMA issuer (leader)
      // A range of kd stages goes into one TMEM accumulator: first the cross products of each
      // stage as it lands (the accumulator is still small), then the hi x hi product of every
      // stage; one commit per range.  The even and odd ranges alternate between two accumulators.
      constexpr uint32_t idesc = idesc_f16(2 * VF_BM, BF_BN, true);
      constexpr int pa_of[5] = {1, 0, 2, 0, 1};   // (A part, B part) of the products before hi x hi
      constexpr int pb_of[5] = {1, 2, 0, 1, 0};
      const uint32_t rdone_bar = smem_u32(rdone);
      const uint64_t desc0 = sdesc_kmajor_sw64(0);
      bool alive = true;
      for (int r = 0; r < n_ranges && alive; ++r) {
        const int it0 = r * kd, it1 = min(n_it, it0 + kd);
        const int b = r & 1, u = r >> 1;
        const uint32_t d_tmem = tmem + b * BF_BN;
        if (u >= 1 && !mbar_spin_warp(&d_free[b], (u - 1) & 1, abort_flag, args.err, DEV_ERR_TIMEOUT_VF)) break;
        for (int it = it0; it < it1; ++it) {
          const int s = it % BF_STAGES;
          if (!(alive = mbar_spin_warp(&full[s], (it / BF_STAGES) & 1, abort_flag, args.err, DEV_ERR_TIMEOUT_VF))) break;
          tc_fence_after();
          const uint64_t sa = desc0 + ((smem_base + s * BF_STAGE) >> 4);
          const uint64_t sb = sa + (BF_PARTS * BF_A_TILE >> 4);
#pragma unroll
          for (int p = 0; p < 5; ++p)
#pragma unroll
            for (int ks = 0; ks < 2; ++ks)
              tc_mma_f16_pair(d_tmem, sa + ((pa_of[p] * BF_A_TILE + ks * 32) >> 4),
                              sb + ((pb_of[p] * BF_B_TILE + ks * 32) >> 4), idesc,
                              it == it0 && p == 0 && ks == 0 ? 0u : 1u);
        }
        if (!alive) break;
        for (int it = it0; it < it1; ++it) {
          const uint64_t sa = desc0 + ((smem_base + (it % BF_STAGES) * BF_STAGE) >> 4);
          const uint64_t sb = sa + (BF_PARTS * BF_A_TILE >> 4);
#pragma unroll
          for (int ks = 0; ks < 2; ++ks) tc_mma_f16_pair(d_tmem, sa + 2 * ks, sb + 2 * ks, idesc);
        }
        tc_commit_pair(rdone_bar + 8 * (r % NRB));
      }
      tc_commit_pair_local(smem_u32(fin_bar));
      int zero = 0;
      mbar_wait(fin_bar, 0, reinterpret_cast<volatile int*>(&zero), args.err, DEV_ERR_TIMEOUT_VF);
    }
  } else {
    // ------------------------------------------------------------------ range drains and epilogue
    const int quarter = warp & 3;
    const int half = (warp - 2) >> 2;
    const uint32_t lane_base = static_cast<uint32_t>(quarter * 32) << 16;
    const uint32_t c_base = static_cast<uint32_t>(half * BF_HC);
    const uint32_t free_bar = cluster_addr(&d_free[0], 0);
    float S[BF_HC];
#pragma unroll
    for (int k = 0; k < BF_HC; ++k) S[k] = 0.0f;
    int nflush = 0;
    auto flush_sums = [&]() {
      double* acc = args.Vacc + (static_cast<int64_t>(split) * args.n_cta + args.cta0 + blockIdx.x) * VF_BM * BF_BN +
                    static_cast<int64_t>(c_base) * VF_BM + quarter * 32 + lane;
      if (valid) {
        if (nflush == 0) {
#pragma unroll
          for (int k = 0; k < BF_HC; ++k) acc[k * VF_BM] = static_cast<double>(S[k]);
        } else {
#pragma unroll
          for (int k = 0; k < BF_HC; ++k) red_add_f64(acc + k * VF_BM, static_cast<double>(S[k]));
        }
      }
#pragma unroll
      for (int k = 0; k < BF_HC; ++k) S[k] = 0.0f;
      ++nflush;
    };
    bool ok = true;
    for (int r = 0; r < n_ranges; ++r) {
      const int b = r & 1;
      // one lane waits, suspended: the board's power is better spent on the MMAs
      if (lane == 0) ok = mbar_wait(&rdone[r % NRB], (r / NRB) & 1, abort_flag, args.err, DEV_ERR_TIMEOUT_VF);
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) break;
      tc_fence_after();
      const uint32_t src = tmem + lane_base + b * BF_BN + c_base;
#pragma unroll
      for (int c = 0; c < BF_HC; c += 16) {
        uint32_t d0[16];
        tmem_ld_x16(src + c, d0);
        tmem_wait_ld();
        if (c + 16 == BF_HC) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(free_bar + 8 * b);
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) S[c + k] += __uint_as_float(d0[k]);
      }
      if (args.flush > 0 && (r + 1) % args.flush == 0) flush_sums();
    }
    if (args.flush > 0) {
      if (ok && n_ranges % args.flush != 0) flush_sums();
    } else {
      const int row = quarter * 32 + lane;
      const int64_t il = static_cast<int64_t>(ib) + row;
      const int pq0 = t.n_tile * BF_BN + static_cast<int>(c_base);
      if (ok && valid && !*abort_flag && il < args.n_i && n_it > 0) {
        float* Vz = args.V + split * v_slice(args.gcp, args.n_orb);
#pragma unroll
        for (int k = 0; k < BF_HC; ++k) {
          const int pq = pq0 + k;
          if (pq < args.n_pair) {
            const int p = __ldg(args.pair_p + pq), q = __ldg(args.pair_q + pq);
            const float v = ldexpf(S[k] * args.unscale_g, -__ldg(args.colexp + pq));
            Vz[v_index(il, p, q, x, args.n_orb)] = v;
            Vz[v_index(il, q, p, x, args.n_orb)] = v;
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync();  // the pair's MMAs, loads and remote arrivals are done
  if (warp == 0) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc_pair(tmem, 512);
  }
}

// =================================================================== finalize kernels
// V from the FP64 accumulator of the GEMM: one CTA per (tile, split, 32 columns), thread = tile row; the tile
// order is the GEMM's grouped order.
constexpr int FIN_COLS = 32;
template <int BN>
__global__ void __launch_bounds__(VF_BM) vfield_finalize_kernel(const VfieldArgs args) {
  const int m_tiles = 3 * args.mt_per_x;
  const TileXY t = pair_tile(blockIdx.x, m_tiles, args.n_tiles);
  if (t.m_tile >= m_tiles) return;
  const int x = t.m_tile / args.mt_per_x;
  const int row = threadIdx.x;
  const int64_t il = static_cast<int64_t>(t.m_tile - x * args.mt_per_x) * VF_BM + row;
  if (il >= args.n_i) return;
  const double* acc = args.Vacc + (static_cast<int64_t>(blockIdx.y) * gridDim.x + blockIdx.x) * VF_BM * BN + row;
  float* v = args.V + blockIdx.y * v_slice(args.gcp, args.n_orb);
  const int ncol = min(BN, args.n_pair - t.n_tile * BN);
  const int c1 = min(ncol, static_cast<int>(blockIdx.z + 1) * FIN_COLS);
#pragma unroll 4
  for (int c = blockIdx.z * FIN_COLS; c < c1; ++c) {
    const int pq = t.n_tile * BN + c;
    const int p = __ldg(args.pair_p + pq), q = __ldg(args.pair_q + pq);
    const float val =
        ldexpf(static_cast<float>(acc[static_cast<int64_t>(c) * VF_BM]) * args.unscale_g, -__ldg(args.colexp + pq));
    v[v_index(il, p, q, x, args.n_orb)] = val;
    v[v_index(il, q, p, x, args.n_orb)] = val;
  }
}

// M[pq][rs] += tile sum * 2^-(exp_a[pq] + exp_b[rs]) for one tile of the step (d) GEMM (mode 1);
// one CTA per tile and slab of 32 columns (each M element is owned by one), through shared memory: read column-major from the tile sums (thread = row), added row-major into M (warp =
// row, lane = column), both coalesced.
template <int BN>
__global__ void __launch_bounds__(VF_BM) assemble_finalize_kernel(const VfieldArgs args) {
  __shared__ double slab[32][VF_BM + 1];
  const int m_tiles = (args.rows_a + VF_BM - 1) / VF_BM;
  const TileXY t = pair_tile(blockIdx.x, m_tiles, args.n_tiles);
  if (t.m_tile >= m_tiles) return;
  const double* acc = args.Vacc + static_cast<int64_t>(blockIdx.x) * VF_BM * BN;
  const int64_t slice = static_cast<int64_t>(gridDim.x) * VF_BM * BN;
  const int ncol = min(BN, args.n_pair - t.n_tile * BN);
  const int row0 = t.m_tile * VF_BM, col0 = t.n_tile * BN;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c0 = blockIdx.z * FIN_COLS;
#pragma unroll
  for (int c = 0; c < 32; c += 8) {
    double v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k)
      v[k] = c0 + c + k < ncol ? acc[static_cast<int64_t>(c0 + c + k) * VF_BM + threadIdx.x] : 0.0;
    for (int z = 1; z < args.slices; ++z)
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (c0 + c + k < ncol) v[k] += acc[z * slice + static_cast<int64_t>(c0 + c + k) * VF_BM + threadIdx.x];
#pragma unroll
    for (int k = 0; k < 8; ++k) slab[c + k][threadIdx.x] = v[k];
  }
  __syncthreads();
  const int c = c0 + lane;
  if (c >= ncol) return;
  const int eb = __ldg(args.exp_b + col0 + c);
#pragma unroll 4
  for (int r = warp; r < VF_BM; r += VF_BM / 32) {
    if (row0 + r >= args.rows_a) break;
    const int pq = row0 + r;
    const int e = __ldg(args.exp_a + pq) + eb;
    double* m = args.M + static_cast<int64_t>(pq) * args.ldm + col0 + c;
    *m += slab[lane][r] * __longlong_as_double(static_cast<long long>(1023 - e) << 52);
  }
}

// CTAs along x: tiles come in pairs of row tiles.
unsigned tile_ctas(const VfieldArgs& a) {
  const int m = a.mode == 0 ? 3 * a.mt_per_x : (a.rows_a + VF_BM - 1) / VF_BM;
  return static_cast<unsigned>((m + 1) / 2 * 2 * a.n_tiles);
}

// CTAs per launch of a GEMM of n CTAs along x.  The CTAs resident at one time stream the same panels of A and
// B and meet in L2 only while they are at about the same k.  Nothing keeps them there: each new tile starts when
// some other one ends, and after ten waves of the N = 120 build the starts are spread over a third of a tile's time,
// with 58.6 GB read from HBM (1,184 outer points) where the panels of its waves are 17 GB (21 now).  The board is at its power cap, so that
// traffic is paid for in clock rate.  Launches of whole waves line the CTAs up again: step (b) of that build 1,060 -> 925 ms,
// of a piece of the N = 200 build 169 -> 134 ms (one wave a launch; two 134, four 139).  A launch costs a few
// microseconds and the tail of its last wave, so it lasts at least LAUNCH_RANGES ranges of 64 values (2 ms;
// at 376 ranges a tile, eight waves a launch are as fast as all of them in one).  Tiles do not depend on each other.
constexpr int LAUNCH_RANGES = 3000;
int launch_ctas(const VfieldArgs& a, int n, int splits) {
  if (splits > 1 || a.n_sm < 2) return n;
  const int64_t ranges = std::max(1, a.n_kb / 2);
  const int64_t step = (LAUNCH_RANGES + ranges - 1) / ranges * (a.n_sm & ~1);
  return static_cast<int>(std::min<int64_t>(std::max(n, 1), step));
}

}  // namespace

int chain_slices(const VfieldArgs& a, int* kb_per_slice) {
  *kb_per_slice = a.n_kb;
  if (a.mode != 1 || a.n_kb % a.kd || a.kd < 2) return 1;
  int flushes = 0;
  const int z = chain_slices(a.n_kb / a.kd, a.flush, 2 * std::max(1, a.xper / (2 * a.kd)), XB_HC,
                             static_cast<int>(tile_ctas(a) / 2), std::max(1, a.n_sm / 2), &flushes);
  if (z > 1) *kb_per_slice = flushes * a.flush * a.kd;
  return z;
}

bool vfield_tc_supported(int n_nuc) { return n_nuc >= 1 && n_nuc <= 8; }

int launch_vfield_tc(const CUtensorMap* tm_g, const CUtensorMap* tm_rho, const CUtensorMap* tm_rho16,
                     const VfieldArgs& a, int parts, int splits, cudaStream_t st) {
  if (a.n_tiles <= 0 || splits <= 0) return 0;
  if (a.mode == 1 ? a.rows_a <= 0 : a.mt_per_x <= 0) return 0;
  dim3 grid(tile_ctas(a), static_cast<unsigned>(splits));
  VfieldArgs w = a;
  w.n_cta = static_cast<int>(grid.x);
  const int step = launch_ctas(a, w.n_cta, splits);
  auto each_launch = [&](auto&& launch) {
    for (w.cta0 = 0; w.cta0 < w.n_cta; w.cta0 += step) {
      grid.x = static_cast<unsigned>(std::min(step, w.n_cta - w.cta0));
      launch(w);
    }
  };
  if (parts == 2) {
    auto kern = a.mode == 1 ? xgemm_kernel<1> : xgemm_kernel<0>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, XB_SMEM);
    each_launch([&](const VfieldArgs& v) { kern<<<grid, XB_THREADS, XB_SMEM, st>>>(*tm_g, *tm_rho, *tm_rho16, v); });
  } else {
    cudaFuncSetAttribute(vfield_bf16_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, BF_SMEM);
    each_launch([&](const VfieldArgs& v) { vfield_bf16_kernel<<<grid, BF_THREADS, BF_SMEM, st>>>(*tm_g, *tm_rho, v); });
  }
  return (w.n_cta + step - 1) / step;
}

void launch_vfield_tc_finalize(const VfieldArgs& a, int parts, int splits, cudaStream_t st) {
  if (a.n_tiles <= 0 || splits <= 0 || a.flush <= 0) return;
  if (a.mode == 1 ? a.rows_a <= 0 : a.mt_per_x <= 0) return;
  dim3 grid(tile_ctas(a), static_cast<unsigned>(splits));
  grid.z = (parts == 2 ? XB_BN : BF_BN) / FIN_COLS;
  if (a.mode == 1) grid.y = 1;  // the kernel adds the slices
  if (a.mode == 1)
    assemble_finalize_kernel<XB_BN><<<grid, VF_BM, 0, st>>>(a);
  else if (parts == 2)
    vfield_finalize_kernel<XB_BN><<<grid, VF_BM, 0, st>>>(a);
  else
    vfield_finalize_kernel<BF_BN><<<grid, VF_BM, 0, st>>>(a);
}

}  // namespace xtc
