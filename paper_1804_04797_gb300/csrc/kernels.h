// Host-side launchers of the CUDA kernels (implemented in the .cu files).
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

#include <cmath>

#include "plan.h"

namespace svk {

struct Mat2 {
  float v[8];  // a, b, c, d as (re, im)
};


// K0: write |0..0> (uniform == false) or the uniform 2^{-n/2} state.  Write-only.
cudaError_t launch_init(float2 *psi, int n, bool uniform, float amp, cudaStream_t st);

// K1/K2/K3 plain tile pass, interpreted: one sweep over all tiles (m qubits) of one pass;
// block: the pass's program in device memory (interp_dev.h), of `bytes` bytes; rk: the
// plan's register slots (2 or 4).
cudaError_t launch_tile_pass(float2 *psi, int n, const unsigned char *block, uint32_t bytes, int m, int rk,
                             cudaStream_t st);
// Largest tile (qubits) of the interpreting plain kernel; the plan-specialised kernels
// take up to svp::kMaxTileBits.
int tile_pass_max_bits();

// K4 fused tensor-core tile pass (tcgen05, split-TF32 or split-FP16).
// r = register qubits of a stage: 5 (tile_bits 12 or 13) or 4 (tile_bits 12); f16: F16x3
// operands, else TF32x3
cudaError_t launch_fused_pass(float2 *psi, int n, const DevPlanView &plan, int pass_index,
                              const svp::DevPass &host_pass, cudaStream_t st, bool f16, int r);
cudaError_t launch_fused_pass_r5(float2 *psi, int n, const DevPlanView &plan, int pass_index,
                                 const svp::DevPass &host_pass, cudaStream_t st, bool f16);
bool fused_supported();

// Per-gate sweeps (K2 one-qubit pair update, K3 diagonal factor on a bit pattern).
cudaError_t launch_gate_1q(float2 *psi, int n, int q, const Mat2 &u, cudaStream_t st);
// amplitudes whose bits under mask equal val are multiplied by (fr + i fi)
cudaError_t launch_gate_diag(float2 *psi, int n, uint64_t mask, uint64_t val, float fr, float fi,
                             cudaStream_t st);

// K5 reductions.  partials: scratch of at least reduce_partials_needed() doubles*2.
int reduce_partials_needed();
cudaError_t launch_norm(const float2 *psi, int n, double *partials, double *out2,
                        cudaStream_t st);
// The second level of launch_norm alone: out2 = the sums of count partial pairs (fixed
// order), e.g. the per-CTA sums a plan kernel's last pass wrote.
cudaError_t launch_norm_final(const double *partials, int count, double *out2, cudaStream_t st);
// out[2j], out[2j+1] = re, im of psi[bits[j]]
cudaError_t launch_gather(const float2 *psi, const uint64_t *bits, int64_t m, double *out,
                          cudaStream_t st);
// out[j] = |psi[bits[j]]|^2
cudaError_t launch_gather_prob(const float2 *psi, const uint64_t *bits, int64_t m, double *out,
                               cudaStream_t st);

// out[(j << t) + l] = A[xa_j + (l << nA)] for l < 2^t.
cudaError_t launch_branch_gather(const float2 *A, int nA, int t, const uint64_t *xa, uint64_t m, float2 *out,
                                 cudaStream_t st);
// K6: out[2j..2j+1] = scale * sum_l A[xa_j + (l << nA)] * B[xb_j + (l << nB)], fp64 (nA < 0: A
// holds what launch_branch_gather wrote).
cudaError_t launch_branch_sum(const float2 *A, int nA, const float2 *B, int nB, int t, const uint64_t *xa,
                              const uint64_t *xb, int m, double scale, double *out, cudaStream_t st);

int device_sm_count();

// Fork of a branch tree: psi[i + (c << n_cur)] = 2^{-(n_new - n_cur)/2} psi[i] for every
// slice c of the branch bits n_cur..n_new-1 (they were |+> until now), in place.
struct ForkScale {
  float hi, lo;  // 2^{-bits/2}: an odd power as the float nearest and the rest
};
inline ForkScale fork_scale(int bits) {
  const double f = std::ldexp(1.0, -(bits / 2)) * ((bits & 1) ? 0.70710678118654752440 : 1.0);
  return ForkScale{(float)f, (float)(f - (double)(float)f)};
}
cudaError_t launch_fork(float2 *psi, int n_cur, int n_new, cudaStream_t st);

// The product of two batched half-states (Eqs. 6-7): A holds 2^t summed branches (bits nA..)
// and above them one bit per branch that a bit of x_B fixes, B likewise.
struct OuterShape {
  int nA = 0, nB = 0, t = 0;
  // x_A's bits in the order of the tiles' columns: those that fix no branch of B (a_free of
  // them, ascending), then those that do; x_B's likewise
  int a_free = 0, b_free = 0;
  uint8_t a_bit[34], b_bit[34];
  // branch bit nA + t + j of A is bit fix_a_by[j] of x_B; nB + t + j of B bit fix_b_by[j] of x_A
  int fix_a = 0, fix_b = 0;
  uint8_t fix_a_by[34], fix_b_by[34];
  // signs (-1)^{x_A bit sign_a[j] * x_B bit sign_b[j]} (crossing CZs that only sign the output)
  int signs = 0;
  uint8_t sign_a[64], sign_b[64];
};

// Full state from the halves: out[x_A + (x_B << nA)] = scale (hi + lo) * the signs * sum over the 2^t
// branches l of A[x_A + (l << nA) + its slice] B[x_B + (l << nB) + its slice] (fp32).  At
// most 2^30 tiles.
cudaError_t launch_outer_sum(const float2 *A, const float2 *B, const OuterShape &shape, float2 scale, float2 *out,
                             cudaStream_t st);
// The same product on the tensor cores (TF32x3, k_outer_tc.cu): at least 7 free bits in
// either half; scratch: outer_sum_tc_scratch bytes of device memory for the operand images;
// err: a device int set non-zero if a bounded wait gave up.
bool outer_sum_tc_supported(const OuterShape &shape);
size_t outer_sum_tc_scratch(const OuterShape &shape);
cudaError_t launch_outer_sum_tc(const float2 *A, const float2 *B, const OuterShape &shape, float2 scale, float2 *out,
                                void *scratch, int *err, cudaStream_t st);

// <a|b> = sum conj(a_i) b_i of two 2^n states: out2 = (re, im), fp64 (partials: 2 *
// reduce_partials_needed() doubles of scratch).
cudaError_t launch_inner(const float2 *a, const float2 *b, int n, double *partials, double *out2, cudaStream_t st);
// The basis state |x>: zero everywhere, 1 at index x.
cudaError_t launch_basis_state(float2 *psi, int n, uint64_t x, cudaStream_t st);

}  // namespace svk
