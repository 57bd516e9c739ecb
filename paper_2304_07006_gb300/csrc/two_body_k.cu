// The two-body transcorrelated integrals K (Theory section, next to the Coulomb integrals V):
//     K_pr^qs = 1/2 <pr| P12 [ lap_1 u + (grad_1 u)^2 + 2 grad_1 u . grad_1 ] |qs>,
//     P12 f(1,2) = f(1,2) + f(2,1),
// on the quadrature grid, for real spatial orbitals.  Written out with the vector pair field
// V_rs(i) = sum_j w_j grad_1 u(r_i, r_j) phi_r(j) phi_s(j) of step (b) and the scalar field
//     W_rs(i) = sum_j w_j F(r_i, r_j) phi_r(j) phi_s(j),   F = lap_1 u + |grad_1 u|^2,
// the f(1,2) part is
//     sum_i [ rho_pq(i) W_rs(i) + 2 psi_pq(i) . V_rs(i) ],  rho_pq = w phi_p phi_q,  psi_pq = w phi_p grad phi_q,
// and the f(2,1) part is the same expression with (pq) and (rs) exchanged (relabel i <-> j; u is
// symmetric).  So with
//     S[pq][rs] = sum_i [ 1/2 rho_pq(i) W_rs(i) + psi_pq(i) . V_rs(i) ]      (pq: all N^2, rs: pairs)
// the integrals are K[p][q][r][s] = S[pq][rs] + S[rs][pq].
//
// Per chunk of outer points: V and W of the chunk as rows [rs][component][i] (V from step (b) in the
// context's precision, W from the same FP64 contraction as the FP64 step (b), with F as the row operand,
// grad64.cu and gemm64_tc.cu), then S accumulates one FP64 contraction over (component, point) whose
// left operand (rho / 2, psi_x) is formed from phi, grad phi and w while it is cut into digits.
#include <algorithm>

#include "xtc_internal.cuh"

namespace xtc {
namespace {

// Index of the pair (min(p,q), max(p,q)) in the packed order p-major, q >= p (the order of the
// pair tables that V and S use).
__device__ __forceinline__ int64_t k_pair(int p, int q, int N) {
  const int a = min(p, q), b = max(p, q);
  return static_cast<int64_t>(a) * N - static_cast<int64_t>(a) * (a - 1) / 2 + (b - a);
}

// K[p][q][r][s] = S[pq][rs] + S[rs][pq]
__global__ void k_unpack_kernel(const double* __restrict__ S, int N, int NP, double* __restrict__ K) {
  const int64_t n2 = static_cast<int64_t>(N) * N;
  const int64_t total = n2 * n2;
  for (int64_t o = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; o < total;
       o += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t left = o / n2, right = o - left * n2;  // (p, q) and (r, s)
    const int p = static_cast<int>(left / N), q = static_cast<int>(left % N);
    const int r = static_cast<int>(right / N), s = static_cast<int>(right % N);
    K[o] = S[left * NP + k_pair(r, s, N)] + S[right * NP + k_pair(p, q, N)];
  }
}

// rows[pq][(1 + x) ncp + i] from V in the layout of v_index; thread = point, a pair and component per CTA row.
__global__ void v_rows_kernel(const float* __restrict__ V, int splits, int n_pair, int n_orb,
                              const int* __restrict__ pair_p, const int* __restrict__ pair_q, int64_t n_i,
                              int64_t gcp, int64_t ncp, double* __restrict__ rows) {
  const int64_t i = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x;
  if (i >= n_i) return;
  const int64_t sstride = v_slice(gcp, n_orb);
  for (int pq = blockIdx.y; pq < n_pair; pq += gridDim.y) {
    const int p = pair_p[pq], q = pair_q[pq];
#pragma unroll
    for (int x = 0; x < 3; ++x) {
      const int64_t idx = v_index(i, p, q, x, n_orb);
      double v = 0.0;
      for (int z = 0; z < splits; ++z) v += static_cast<double>(V[z * sstride + idx]);
      rows[pq * 4 * ncp + (1 + x) * ncp + i] = v;
    }
  }
}

}  // namespace

void launch_v_rows(const float* V, int splits, int n_pair, int n_orb, const int* pair_p, const int* pair_q,
                   int64_t n_i, int64_t gcp, int64_t ncp, double* rows, cudaStream_t st) {
  const dim3 g(static_cast<unsigned>((n_i + 127) / 128), static_cast<unsigned>(std::min(n_pair, 65535)));
  v_rows_kernel<<<g, 128, 0, st>>>(V, splits, n_pair, n_orb, pair_p, pair_q, n_i, gcp, ncp, rows);
}

void launch_k_unpack(const double* S, int n_orb, double* K, int n_sm, cudaStream_t st) {
  const int NP = n_orb * (n_orb + 1) / 2;
  const int64_t n2 = static_cast<int64_t>(n_orb) * n_orb;
  const int64_t blocks = std::min<int64_t>((n2 * n2 + 255) / 256, static_cast<int64_t>(n_sm) * 32);
  k_unpack_kernel<<<static_cast<unsigned>(blocks), 256, 0, st>>>(S, n_orb, NP, K);
}

}  // namespace xtc
