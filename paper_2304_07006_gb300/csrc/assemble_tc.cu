// Step (d) on the tensor cores: the two-body assembly of Appendix B,
//     Delta U(pq|rs) = -sum_i [rho_pq A_rs + V_pq . B_rs + rho_rs A_pq + V_rs . B_pq]
// computed as M += L^T R with L[pq][k] = (rho, Vx, Vy, Vz) and R[rs][k] = (A, Bx, By, Bz) for
// k = (outer point, component); Delta U = -(M + M^T) is formed by the final kernels.
//
// CTA tile 128 x 128, 32-element K stages with both operands TMA-loaded in the 64-byte swizzle,
// three bf16 parts per operand and six split products (i + j <= 2, smallest first).  Warp 0 issues
// the TMA loads, warp 1 the MMAs into one of two TMEM accumulators; every `kd` stages warps 2..17
// add the finished accumulator into a compensated FP32 running sum (sum and error term, Knuth's
// TwoSum, in registers, 32 columns a thread) while the MMA fills the other one, which keeps the tensor-core
// accumulation (truncating at each MMA) to short ranges.  A tcgen05.commit stalls the tensor pipe
// for a few hundred cycles, so each range ends with one commit, whose arrival both frees the
// range's stage slots (the TMA producer counts finished ranges in order) and starts the drain.
// At the end warps 2..17 add sum + error into the FP64 accumulator M in HBM (read-modify-write;
// every tile of M is owned by exactly one CTA).
#include "ptx_sm100.cuh"
#include "xtc_internal.cuh"

namespace xtc {
namespace {

constexpr int PARTS = 3;
constexpr int NPROD = 6;
constexpr int STAGES = 4;
constexpr int A_TILE = AS_BM * 64;
constexpr int B_TILE = AS_BN * 64;
constexpr int STAGE_BYTES = PARTS * (A_TILE + B_TILE);
constexpr int SMEM = STAGES * STAGE_BYTES + 1024 + 256;
constexpr int DRAIN_WARPS = 16;        // four per TMEM lane quarter, a quarter of the columns each
constexpr int THREADS = (2 + DRAIN_WARPS) * 32;
constexpr int HC = AS_BN / 4;          // running-sum columns per drain thread
constexpr int TMEM_COLS = 2 * AS_BN;
static_assert(HC == 32 && TMEM_COLS == 256, "drain columns; TMEM allocation (a power of 2)");
constexpr int NRB = 8;                 // range barriers (range r uses r % NRB)
// a wait for range r must not alias range r + NRB (the producer waits for the range of stage
// k - STAGES before loading stage k)
static_assert(NRB > STAGES, "range barriers");

__device__ __forceinline__ void tmem_ld_x16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}

// *p += s + c in FP64.  The conversions stay beside the access: hoisted out of a row of these, they would not
// fit the registers.
__device__ __forceinline__ void add_f64(double* p, float s, float c) {
  asm volatile(
      "{\n\t.reg .f64 a, b;\n\t"
      "cvt.f64.f32 a, %1;\n\tcvt.f64.f32 b, %2;\n\tadd.rn.f64 a, a, b;\n\t"
      "ld.global.f64 b, [%0];\n\tadd.rn.f64 b, b, a;\n\tst.global.f64 [%0], b;\n\t}" ::"l"(p),
      "f"(s), "f"(c)
      : "memory");
}

__global__ void __launch_bounds__(THREADS, 1)
    assemble_tc_kernel(const __grid_constant__ CUtensorMap tm_L, const __grid_constant__ CUtensorMap tm_R,
                       int n_pair, int ldm, int n_kb, int kd, double* __restrict__ M, int* err) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
  uint64_t* full = bars;                     // [STAGES] the stage's loads landed
  uint64_t* rdone = bars + STAGES;           // [NRB] the MMAs of range r (r % NRB) completed
  uint64_t* d_free = bars + STAGES + NRB;    // [2] the drains released accumulator b
  uint64_t* fin_bar = bars + STAGES + NRB + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + STAGES + NRB + 3);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;  // warp: uniform
  const int m_tile = blockIdx.x, n_tile = blockIdx.y;
  const int n_ranges = (n_kb + kd - 1) / kd;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) mbar_init(&full[s], 1);
    for (int r = 0; r < NRB; ++r) mbar_init(&rdone[r], 1);
    for (int b = 0; b < 2; ++b) mbar_init(&d_free[b], DRAIN_WARPS);
    mbar_init(fin_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
    tma_prefetch_desc(&tm_L);
    tma_prefetch_desc(&tm_R);
  }
  if (warp == 0) {
    tmem_alloc(tmem_slot, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t smem_base = smem_u32(smem);

  if (warp == 0) {
    if (lane == 0) {
      int seen = 0;  // ranges known to have completed (their slots are free again)
      int issued_end = 0;
      for (int kb = 0; kb < n_kb; ++kb) {
        const int s = kb % STAGES;
        if (kb >= STAGES) {
          const int need = (kb - STAGES) / kd;  // range holding the slot's previous stage
          bool ok = true;
          for (; seen <= need && ok; ++seen)
            ok = mbar_wait(&rdone[seen % NRB], (seen / NRB) & 1, abort_flag, err, DEV_ERR_TIMEOUT_AS);
          if (!ok) break;
        }
        mbar_arrive_expect_tx(&full[s], STAGE_BYTES);
        uint8_t* st = smem + s * STAGE_BYTES;
        for (int p = 0; p < PARTS; ++p) {
          tma_load_3d(st + p * A_TILE, &tm_L, &full[s], kb * AS_BK, m_tile * AS_BM, p);
          tma_load_3d(st + PARTS * A_TILE + p * B_TILE, &tm_R, &full[s], kb * AS_BK, n_tile * AS_BN, p);
        }
        issued_end = kb + 1;
      }
      int zero = 0;
      for (int kb = max(0, issued_end - STAGES); kb < issued_end; ++kb)
        mbar_wait(&full[kb % STAGES], (kb / STAGES) & 1, reinterpret_cast<volatile int*>(&zero), err,
                  DEV_ERR_TIMEOUT_AS);
    }
  } else if (warp == 1) {
    // The whole warp runs the loop, so that descriptors stay in uniform registers: one thread encoding and
    // spilling them took 4,350 cycles for the 24 MMAs of a range (1,536 cycles of tensor pipe), and that bound the kernel.
    // Step (d) of a water-sized build (58 orbitals, 40,000 points): 17.9 -> 11.4 ms.
    constexpr uint32_t idesc = idesc_f16(AS_BM, AS_BN, true);
    // small cross products first, hi x hi last, over all stages of a range (the early
    // truncations then act on a small accumulator)
    constexpr int pa_of[5] = {1, 0, 2, 0, 1};
    constexpr int pb_of[5] = {1, 2, 0, 1, 0};
    const uint64_t desc0 = sdesc_kmajor_sw64(0);
    const uint32_t rdone_bar = smem_u32(rdone);
    bool alive = true;
    for (int r = 0; r < n_ranges && alive; ++r) {
      const int kb0 = r * kd, kb1 = min(n_kb, kb0 + kd);
      const int b = r & 1, u = r >> 1;
      const uint32_t d = tmem + b * AS_BN;
      if (u >= 1 && !mbar_spin_warp(&d_free[b], (u - 1) & 1, abort_flag, err, DEV_ERR_TIMEOUT_AS)) break;
      // cross products of each stage as it lands, then the hi x hi products of the range
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!(alive = mbar_spin_warp(&full[kb % STAGES], (kb / STAGES) & 1, abort_flag, err, DEV_ERR_TIMEOUT_AS))) break;
        tc_fence_after();
        const uint64_t sa = desc0 + ((smem_base + (kb % STAGES) * STAGE_BYTES) >> 4), sb = sa + (PARTS * A_TILE >> 4);
#pragma unroll
        for (int p = 0; p < NPROD - 1; ++p)
#pragma unroll
          for (int ks = 0; ks < 2; ++ks)
            tc_mma_f16_warp(d, sa + ((pa_of[p] * A_TILE + ks * 32) >> 4), sb + ((pb_of[p] * B_TILE + ks * 32) >> 4),
                            idesc, kb == kb0 && p == 0 && ks == 0 ? 0u : 1u);
      }
      if (!alive) break;
      for (int kb = kb0; kb < kb1; ++kb) {
        const uint64_t sa = desc0 + ((smem_base + (kb % STAGES) * STAGE_BYTES) >> 4), sb = sa + (PARTS * A_TILE >> 4);
#pragma unroll
        for (int ks = 0; ks < 2; ++ks) tc_mma_f16_warp(d, sa + 2 * ks, sb + 2 * ks, idesc, 1u);
      }
      tc_commit_warp(rdone_bar + 8 * (r % NRB));
    }
    tc_commit_warp(smem_u32(fin_bar));
    int zero = 0;
    mbar_wait(fin_bar, 0, reinterpret_cast<volatile int*>(&zero), err, DEV_ERR_TIMEOUT_AS);
  } else {
    const int quarter = warp & 3;               // TMEM lanes 32*quarter .. +31 (hardware rule)
    const int c_base = ((warp - 2) >> 2) * HC;  // columns c_base .. +HC-1
    const uint32_t my = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + c_base;
    float S[HC], C[HC];
#pragma unroll
    for (int k = 0; k < HC; ++k) S[k] = C[k] = 0.0f;
    bool ok = true;
#pragma unroll 1
    for (int r = 0; r < n_ranges; ++r) {
      const int b = r & 1;
      // one lane waits, suspended (the board's power is better spent on the MMAs)
      if (lane == 0) ok = mbar_wait(&rdone[r % NRB], (r / NRB) & 1, abort_flag, err, DEV_ERR_TIMEOUT_AS);
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) break;
      tc_fence_after();
#pragma unroll
      for (int c0 = 0; c0 < HC; c0 += 16) {
        uint32_t d[16];
        tmem_ld_x16(my + b * AS_BN + c0, d);
        tmem_wait_ld();
        if (c0 + 16 == HC) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&d_free[b]);
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          // TwoSum: s1 + e == x + y exactly (the first range gives s1 = y, e = 0)
          const float x = S[c0 + k], y = __uint_as_float(d[k]);
          const float s1 = __fadd_rn(x, y);
          const float yp = __fsub_rn(s1, x);
          const float xp = __fsub_rn(s1, yp);
          const float e = __fadd_rn(__fsub_rn(x, xp), __fsub_rn(y, yp));
          S[c0 + k] = s1;
          C[c0 + k] = __fadd_rn(C[c0 + k], e);
        }
      }
    }
    const int row = m_tile * AS_BM + quarter * 32 + lane;
    const int col0 = n_tile * AS_BN + c_base;
    if (ok && !*abort_flag && row < n_pair && n_kb > 0 && col0 < n_pair) {
      double* dst = M + static_cast<int64_t>(row) * ldm + col0;
#pragma unroll
      for (int k = 0; k < HC; ++k) add_f64(dst + k, S[k], C[k]);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

}  // namespace

void launch_assemble_tc(const CUtensorMap* tm_L, const CUtensorMap* tm_R, int n_pair, int kdim, int kd, double* M,
                        int* err, cudaStream_t st) {
  // M has row stride m_stride(n_pair) so every 32-column group of a tile is in bounds
  const int ldm = static_cast<int>(m_stride(n_pair));
  cudaFuncSetAttribute(assemble_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
  dim3 grid((n_pair + AS_BM - 1) / AS_BM, (n_pair + AS_BN - 1) / AS_BN);
  assemble_tc_kernel<<<grid, THREADS, SMEM, st>>>(*tm_L, *tm_R, n_pair, ldm, kdim / AS_BK, kd, M, err);
}

}  // namespace xtc
