// K6: fp64 branch sum of the cut decomposition (§2, Fig. 2 and Eq. 1).
//
// The two halves are stored as batched states: A[x_A + (l << nA)] is amplitude x_A of
// branch l of half A (and likewise B), so branch l of every half-state is one slice of
// a (nA + t)-qubit vector.  For each requested bitstring j one CTA forms
// sum_l A[xa_j, l] * B[xb_j, l] in fp64 with a fixed reduction tree (deterministic).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "kernels.h"

namespace svk {
namespace {

constexpr int kBlock = 256;

__global__ void branch_sum_kernel(const float2 *__restrict__ A, int nA, const float2 *__restrict__ B, int nB,
                                  int t, const uint64_t *__restrict__ xa, const uint64_t *__restrict__ xb,
                                  double scale, double *__restrict__ out) {
  const int j = blockIdx.x;
  const uint64_t branches = 1ull << t;
  // (nA < 0: A holds branch_gather_kernel's slices)
  const uint64_t a0 = nA < 0 ? (uint64_t)j << t : xa[j], b0 = xb[j];
  const int sa = nA < 0 ? 0 : nA;
  double sr = 0.0, si = 0.0;
  for (uint64_t l = threadIdx.x; l < branches; l += blockDim.x) {
    const float2 a = A[a0 + (l << sa)];
    const float2 b = B[b0 + (l << nB)];
    sr += (double)a.x * b.x - (double)a.y * b.y;
    si += (double)a.x * b.y + (double)a.y * b.x;
  }
  __shared__ double rr[kBlock], ri[kBlock];
  rr[threadIdx.x] = sr;
  ri[threadIdx.x] = si;
  __syncthreads();
  for (int h = kBlock / 2; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) {
      rr[threadIdx.x] += rr[threadIdx.x + h];
      ri[threadIdx.x] += ri[threadIdx.x + h];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[2 * j] = rr[0] * scale;
    out[2 * j + 1] = ri[0] * scale;
  }
}

// The 2^t branch amplitudes of each bitstring's half index xa[j], one bitstring after the other.
__global__ void branch_gather_kernel(const float2 *__restrict__ A, int nA, int t, const uint64_t *__restrict__ xa,
                                     uint64_t count, float2 *__restrict__ out) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < count; i += (uint64_t)gridDim.x * blockDim.x)
    out[i] = A[xa[i >> t] + ((i & ((1ull << t) - 1)) << nA)];
}

// The tensor form of the same sum (§2, Eqs. 6-7: the full state is a sum over branches
// of outer products phi_l (x) xi_l): out[x_A + (x_B << nA)] = scale * sum_l
// A_l[x_A] * B_l[x_B], a complex matrix product (2^nB x 2^t) * (2^t x 2^nA), times the signs
// (-1)^{x_a x_b} of absorbed CZs.  fp32 accumulation.
//
// Only the fully decomposed CZs are summed over.  An implicitly decomposed one (§2.1) has its
// branch fixed by an output bit: one on a qubit of A by a bit of x_A, which selects the slice
// of B, and the other way round.  So the tiles are taken over the columns (rows) that agree
// in those bits, and every tile is a product over 2^t branches of its own slices.
//
// Bound by the write of the state up to about 2^4 branches, above that by the FP32 pipe (8 *
// 2^t flops an amplitude).  128 x 64 outputs per CTA of 256 threads; a thread holds 4 rows
// of 4 pairs of columns as packed accumulators (re, re') and (im, im'), so that a row's factor
// (bx, bx), (by, by) and a pair's (ax, ax'), (ay, ay') -- 8 reads of 16 bytes, both expanded
// once on their way into shared memory -- feed 64 packed FMAs, and a pair of neighbours is
// one 16-byte store.  Two CTAs an SM (128 registers a thread): one stores while the other
// computes (persistent CTAs that fetch the next tile while they store measured 1.38 ms).
// 28 qubits on one GB300, 4x7 lattice of depth 10 (6 expanded CZs, 2 of them implicit): every
// expanded CZ summed over, 4 x 4 outputs a thread and scalar FMAs 3.1 ms (2^6 branches) and
// 6.2 ms (2^7); these tiles 2.8 and 5.2 ms; with the implicit branches fixed by tile 1.08 ms
// (2^4) and 1.45 ms (2^5); the write alone takes 0.32 ms.
constexpr int kColsA = 128, kRowsB = 64, kStep = 8;

__device__ __forceinline__ uint64_t warp_or(uint64_t x) {
  return (uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(x >> 32)) << 32 |
         __reduce_or_sync(0xffffffffu, (uint32_t)x);
}

// SCALED: signs, or a scale with a lo part.
template <bool SCALED>
__global__ void __launch_bounds__(256, 2) outer_sum_kernel(const float2 *__restrict__ A, const float2 *__restrict__ B,
                                                           const OuterShape S, float2 scale, int tiles_a_log2,
                                                           float2 *__restrict__ out) {
  __shared__ float4 As[2][kStep][kColsA / 2], Bs[2][kStep][kRowsB];
  __shared__ uint64_t col_at[kColsA], row_at[kRowsB];  // x_A of the tile's columns, x_B of its rows
  // 2^t branches (t up to 33: their number takes 34 bits) in steps of kStep or fewer
  const uint32_t steps = 1u << max(S.t - 3, 0), last = steps - 1;
  const int per_step = 1 << min(S.t, 3);
  const int nA = S.nA, nB = S.nB, tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, lane = tid & 31;
  const uint32_t ct = blockIdx.x & ((1u << tiles_a_log2) - 1), rt = blockIdx.x >> tiles_a_log2;
  // the index bits in the order of S.a_bit and S.b_bit, a slice's (the last ones) above the tiles
  const int ca_bits = min(S.a_free, 7), rb_bits = min(S.b_free, 6);
  const uint64_t xa0 = warp_or(lane < nA - ca_bits ? (uint64_t)((ct >> lane) & 1u) << S.a_bit[ca_bits + lane] : 0);
  const uint64_t xb0 = warp_or(lane < nB - rb_bits ? (uint64_t)((rt >> lane) & 1u) << S.b_bit[rb_bits + lane] : 0);
  if (tid < kColsA) {
    uint64_t x = xa0;
#pragma unroll
    for (int i = 0; i < 7; ++i) x |= i < ca_bits ? (uint64_t)((tid >> i) & 1) << S.a_bit[i] : 0;
    col_at[tid] = x;
  } else if (tid < kColsA + kRowsB) {
    uint64_t x = xb0;
#pragma unroll
    for (int i = 0; i < 6; ++i) x |= i < rb_bits ? (uint64_t)((tid >> i) & 1) << S.b_bit[i] : 0;
    row_at[tid - kColsA] = x;
  }
  // the slices that the tile's fixed bits select
  const uint64_t off_a = warp_or(lane < S.fix_a ? ((xb0 >> S.fix_a_by[lane]) & 1ull) << (nA + S.t + lane) : 0);
  const uint64_t off_b = warp_or(lane < S.fix_b ? ((xa0 >> S.fix_b_by[lane]) & 1ull) << (nB + S.t + lane) : 0);
  __syncthreads();
  // the thread's share of a step's operands: column tid mod 128 of A in every other branch,
  // row tid mod 64 of B in every fourth
  const int ca = tid & 127, ka = tid >> 7, rb = tid & 63, kb = tid >> 6;
  const bool in_a = ca < (1 << ca_bits), in_b = rb < (1 << rb_bits);
  const float2 *pa = A + off_a + col_at[ca] + ((uint64_t)ka << nA), *pb = B + off_b + row_at[rb] + ((uint64_t)kb << nB);
  const uint64_t step_a = 2ull << nA, step_b = 4ull << nB;
  float2 va[kStep / 2], vb[kStep / 4];
  auto fetch = [&]() {
#pragma unroll
    for (int k = 0; k < kStep / 2; ++k, pa += step_a)
      va[k] = in_a && 2 * k + ka < per_step ? *pa : make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < kStep / 4; ++k, pb += step_b)
      vb[k] = in_b && 4 * k + kb < per_step ? *pb : make_float2(0.f, 0.f);
  };
  float2 re[4][4], im[4][4];  // [row][pair]
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int j = 0; j < 4; ++j) re[r][j] = im[r][j] = make_float2(0.f, 0.f);
  fetch();
  int s = 0;
  for (uint32_t step = 0; step <= last; ++step, s ^= 1) {
#pragma unroll
    for (int k = 0; k < kStep / 2; ++k) {
      float *const p = reinterpret_cast<float *>(&As[s][2 * k + ka][ca >> 1]) + (ca & 1);
      p[0] = va[k].x;
      p[2] = va[k].y;
    }
#pragma unroll
    for (int k = 0; k < kStep / 4; ++k) Bs[s][4 * k + kb][rb] = make_float4(vb[k].x, vb[k].x, vb[k].y, vb[k].y);
    __syncthreads();  // (two buffers: the step before the last has been read by every thread)
    if (step < last) fetch();
#pragma unroll 1  // (unrolled 2, 4, 8 times: 1.10, 1.14, 1.23 ms against 1.08 at 28 qubits, 2^4 branches)
    for (int k = 0; k < per_step; ++k) {
      float4 a[4], b[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) a[j] = As[s][k][16 * j + tx];
#pragma unroll
      for (int r = 0; r < 4; ++r) b[r] = Bs[s][k][16 * r + ty];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float2 bx = make_float2(b[r].x, b[r].y), by = make_float2(b[r].z, b[r].w);
        const float2 ny = make_float2(-b[r].z, -b[r].w);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float2 ax = make_float2(a[j].x, a[j].y), ay = make_float2(a[j].z, a[j].w);
          re[r][j] = __ffma2_rn(ax, bx, __ffma2_rn(ay, ny, re[r][j]));
          im[r][j] = __ffma2_rn(ax, by, __ffma2_rn(ay, bx, im[r][j]));
        }
      }
    }
  }
  // columns 2 tx + 32 j and the next, rows 16 r + ty of the tile
  const bool neighbours = ca_bits > 0 && S.a_bit[0] == 0;
  uint64_t c0[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) c0[j] = col_at[2 * tx + 32 * j];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int row = 16 * r + ty;
    if (row >= (1 << rb_bits)) continue;
    const uint64_t xb = row_at[row];
    float2 *const to = out + (xb << nA);
    uint64_t m = 0;  // bits of x_A whose parity is the row's sign
    if (SCALED)
      for (int j = 0; j < S.signs; ++j) m ^= ((xb >> S.sign_b[j]) & 1ull) << S.sign_a[j];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int col = 2 * tx + 32 * j;
      if (col >= (1 << ca_bits)) continue;
      float4 v = make_float4(re[r][j].x, im[r][j].x, re[r][j].y, im[r][j].y);
      if (SCALED) {
        const uint32_t s0 = (uint32_t)__popcll(m & c0[j]) << 31, s1 = (uint32_t)__popcll(m & col_at[col + 1]) << 31;
        auto scaled = [&](float x, uint32_t sign) {
          return __uint_as_float(__float_as_uint(fmaf(x, scale.x, x * scale.y)) ^ sign);
        };
        v = make_float4(scaled(v.x, s0), scaled(v.y, s0), scaled(v.z, s1), scaled(v.w, s1));
      } else {
        v = make_float4(v.x * scale.x, v.y * scale.x, v.z * scale.x, v.w * scale.x);
      }
      if (neighbours) {
        *reinterpret_cast<float4 *>(to + c0[j]) = v;
      } else {
        to[c0[j]] = make_float2(v.x, v.y);
        if (col + 1 < (1 << ca_bits)) to[col_at[col + 1]] = make_float2(v.z, v.w);
      }
    }
  }
}

// A fork of the branch tree: the first 2^n_cur amplitudes (every branch bit above them
// still in |+>) replicated into all 2^(n_new - n_cur) slices of new branch bits, each
// times 2^{-(n_new - n_cur)/2} (the H that put those bits in |+>): psi[i + (c << n_cur)]
// = f psi[i].  Two amplitudes per 16-byte vector; f applied as hi + lo (one rounding).
__global__ void fork_kernel(float4 *__restrict__ psi, uint64_t pairs, int copies_log2, int n_cur, float f_hi,
                            float f_lo) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < pairs; i += stride) {
    float4 v = psi[i];
    v.x = fmaf(v.x, f_hi, v.x * f_lo);
    v.y = fmaf(v.y, f_hi, v.y * f_lo);
    v.z = fmaf(v.z, f_hi, v.z * f_lo);
    v.w = fmaf(v.w, f_hi, v.w * f_lo);
    for (uint64_t c = 0; c < (1ull << copies_log2); ++c) psi[i + (c << (n_cur - 1))] = v;
  }
}

}  // namespace

cudaError_t launch_fork(float2 *psi, int n_cur, int n_new, cudaStream_t st) {
  if (n_new <= n_cur) return cudaSuccess;
  if (n_cur < 1) return cudaErrorInvalidValue;
  const int k = n_new - n_cur;
  const ForkScale f = fork_scale(k);
  const uint64_t pairs = 1ull << (n_cur - 1);
  uint64_t grid = (pairs + 255) / 256;
  const uint64_t cap = (uint64_t)device_sm_count() * 16;
  if (grid > cap) grid = cap;
  fork_kernel<<<(unsigned)grid, 256, 0, st>>>(reinterpret_cast<float4 *>(psi), pairs, k, n_cur, f.hi, f.lo);
  return cudaGetLastError();
}

cudaError_t launch_outer_sum(const float2 *A, const float2 *B, const OuterShape &S, float2 scale, float2 *out,
                             cudaStream_t st) {
  const int ta = S.nA - std::min(S.a_free, 7), tb = S.nB - std::min(S.b_free, 6);  // log2 of the tiles
  if (S.nA < 1 || S.nB < 1 || ta + tb > 30) return cudaErrorInvalidValue;
  const bool scaled = S.signs > 0 || scale.y != 0.f;
  (scaled ? outer_sum_kernel<true> : outer_sum_kernel<false>)<<<1u << (ta + tb), 256, 0, st>>>(A, B, S, scale, ta, out);
  return cudaGetLastError();
}

cudaError_t launch_branch_gather(const float2 *A, int nA, int t, const uint64_t *xa, uint64_t m, float2 *out,
                                 cudaStream_t st) {
  const uint64_t count = m << t;
  if (count == 0) return cudaSuccess;
  const unsigned grid = (unsigned)std::min<uint64_t>((count + kBlock - 1) / kBlock, (uint64_t)device_sm_count() * 8);
  branch_gather_kernel<<<grid, kBlock, 0, st>>>(A, nA, t, xa, count, out);
  return cudaGetLastError();
}

cudaError_t launch_branch_sum(const float2 *A, int nA, const float2 *B, int nB, int t, const uint64_t *xa,
                              const uint64_t *xb, int m, double scale, double *out, cudaStream_t st) {
  if (m <= 0) return cudaSuccess;
  branch_sum_kernel<<<m, kBlock, 0, st>>>(A, nA, B, nB, t, xa, xb, scale, out);
  return cudaGetLastError();
}

}  // namespace svk
