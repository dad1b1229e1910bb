// The tensor form of the cut decomposition on the tcgen05 tensor cores (Eqs. 6-7):
//     psi_AB[x_A + 2^nA x_B] = scale * sum_l A_l[x_A] B_l[x_B],
// i.e. the complex product Psi = Bm Am^T of the half-states' branch matrices Bm (2^nB x L)
// and Am (2^nA x L), L = 2^t summed branches, as one real GEMM with K = 2L (where a branch is
// fixed by an output bit, one for every combination of slices, the rows and columns taken
// in OuterShape's order):
//     D[x_B, 2 x_A + o] = sum_{l, c} Aop[x_B, 2l + c] Bop[2 x_A + o, 2l + c],
//     Aop[x_B, 2l + c] = (Re, Im)_c B_l[x_B],
//     Bop[2 x_A, 2l + c] = (Re A_l[x_A], -Im A_l[x_A])_c,  Bop[2 x_A + 1, 2l + c] = (Im, Re)_c,
// so a row of D is a contiguous run of output amplitudes (re, im interleaved).  TF32x3:
// each operand is split into hi + lo (nearest TF32 values) and D = Ahi Bhi + Ahi Blo +
// Alo Bhi is accumulated in fp32 in tensor memory (the lo*lo term is ~2^-22 relative).
//
// A prep kernel writes the split operands as images in the MMA's shared-memory layout
// (K-major, no swizzle: 8-row x 16-byte core matrices), one contiguous block per (slice, row
// tile, 32-wide K chunk), so a CTA fetches each with one bulk copy.  The GEMM kernel is
// persistent (two CTAs per SM: one stores its tile while the other computes): per output
// tile of 128 x 128 amplitudes it loads the blocks of every K chunk, one thread issues the
// 3 x 4 MMAs (M = 128, N = 256, K = 8) per chunk, and the warps move D from tensor memory
// through shared memory to HBM in whole 128-byte runs of the state.  All waits are bounded.
#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.h"

namespace svk {
namespace {

constexpr int kRows = 128;                         // output rows (x_B) per tile
constexpr int kCols = 128;                         // output amplitudes (x_A) per tile
constexpr int kKc = 32;                            // real K per chunk
constexpr uint32_t kABlock = kRows * kKc * 4;      // one part of an A block (16 KB)
constexpr uint32_t kBBlock = 2 * kCols * kKc * 4;  // one part of a B block (32 KB)
constexpr uint32_t kSmem = 2 * kABlock + 2 * kBBlock;
constexpr unsigned long long kWaitNs = 1000000000ull;
// kind::tf32, D fp32, A and B K-major, N = 256, M = 128
constexpr uint32_t kIdesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(256 >> 3) << 17) | (8u << 24);

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Byte offset of (row, k) in a block of `rows` x 32 tf32 values, K-major without swizzle:
// core matrices of 8 rows x 4 values (16 B), K-adjacent ones 128 B apart, 8-row groups
// 1024 B apart.
__host__ __device__ __forceinline__ uint32_t blk_off(uint32_t row, uint32_t k) {
  return ((row >> 3) * (kKc / 4) + (k >> 2)) * 128u + (row & 7u) * 16u + (k & 3u) * 4u;
}

__device__ __forceinline__ float tf32_rn(float x) {
  return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xFFFFE000u);
}

// Index bits of x spread over a half's qubits in OuterShape's order.
__device__ __forceinline__ uint64_t spread(uint64_t i, const uint8_t *bit, int n) {
  uint64_t x = 0;
  for (int k = 0; k < n; ++k) x |= ((i >> k) & 1ull) << bit[k];
  return x;
}

// Operand images.  Aop: slice s of B, row tile rt, chunk kc at (((s * rtiles + rt) * kch + kc) *
// 2 + part) * kABlock; Bop likewise with A, its column tiles and kBBlock.  One thread per
// (slice, row, k) of each operand.  FIXED: as below.
template <bool FIXED>
__global__ void outer_prep_kernel(const float2 *__restrict__ A, const float2 *__restrict__ B, const OuterShape S,
                                  int kch, unsigned char *__restrict__ aimg, unsigned char *__restrict__ bimg) {
  const uint64_t L = 1ull << S.t, K = (uint64_t)kch * kKc;
  const uint64_t na = 1ull << S.nA, nb = 1ull << S.nB;
  const uint64_t nA_ops = (nb << S.fix_b) * K, nB_ops = 2 * (na << S.fix_a) * K;
  for (uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nA_ops + nB_ops;
       e += (uint64_t)gridDim.x * blockDim.x) {
    float v;
    unsigned char *dst;
    uint32_t blk;
    if (e < nA_ops) {  // Aop[row, k] of slice row / nb
      const uint64_t row = e / K, k = e % K, l = k >> 1, slice = FIXED ? row >> S.nB : 0;
      const uint64_t xb = FIXED ? spread(row & (nb - 1), S.b_bit, S.nB) : row;
      const float2 z = l < L ? B[xb + (l << S.nB) + (slice << (S.nB + S.t))] : make_float2(0.f, 0.f);
      v = (k & 1) ? z.y : z.x;
      const uint64_t rt = row / kRows, kc = k / kKc;
      dst = aimg + (rt * kch + kc) * 2 * kABlock;
      blk = kABlock;
      const uint32_t o = blk_off((uint32_t)(row % kRows), (uint32_t)(k % kKc));
      const float h = tf32_rn(v);
      *reinterpret_cast<float *>(dst + o) = h;
      *reinterpret_cast<float *>(dst + blk + o) = tf32_rn(v - h);
    } else {  // Bop[n, k], n = 2 column + o, of slice column / na
      const uint64_t f = e - nA_ops, n = f / K, k = f % K, l = k >> 1, slice = FIXED ? (n >> 1) >> S.nA : 0;
      const uint64_t xa = FIXED ? spread((n >> 1) & (na - 1), S.a_bit, S.nA) : n >> 1;
      const float2 z = l < L ? A[xa + (l << S.nA) + (slice << (S.nA + S.t))] : make_float2(0.f, 0.f);
      const bool im_out = n & 1, im_in = k & 1;
      v = !im_out ? (im_in ? -z.y : z.x) : (im_in ? z.x : z.y);
      const uint64_t ct = n / (2 * kCols), kc = k / kKc;
      dst = bimg + (ct * kch + kc) * 2 * kBBlock;
      blk = kBBlock;
      const uint32_t o = blk_off((uint32_t)(n % (2 * kCols)), (uint32_t)(k % kKc));
      const float h = tf32_rn(v);
      *reinterpret_cast<float *>(dst + o) = h;
      *reinterpret_cast<float *>(dst + blk + o) = tf32_rn(v - h);
    }
  }
}

__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);
  d |= (uint64_t)(128 >> 4) << 16;   // K-adjacent core matrices
  d |= (uint64_t)(1024 >> 4) << 32;  // 8-row groups
  d |= (uint64_t)1 << 46;
  return d;
}
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t a, uint64_t b, uint32_t acc) {
  asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n"
               ::"r"(d), "l"(a), "l"(b), "r"(kIdesc), "r"(acc));
}
__device__ __forceinline__ bool mbar_try(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile("{\n .reg .pred P1;\n mbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n selp.b32 %0, 1, 0, P1;\n}\n"
               : "=r"(ok)
               : "r"(smem_u32(bar)), "r"(parity)
               : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
  if (mbar_try(bar, parity)) return true;
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  do {
    if (mbar_try(bar, parity)) return true;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  } while (t - t0 < kWaitNs);
  return false;
}

// FIXED: some branches are fixed by output bits, so that a tile's rows and columns lie in
// OuterShape's order (else in the state's: one address per row).  SCALED: with signs, or a scale
// with a lo part.  A product that needs neither (every expanded CZ summed over) keeps to one
// multiplication a value and a running address, and its operands' images to the state's order.
// Both kernels with one form for all / with these, us at 28 qubits on one GB300: 2^7 branches
// summed 1415 / 1355, 2^4 and three signs 696 / 640, 2^5 and two more fixed 644 / 645.
template <bool FIXED, bool SCALED>
__global__ void __launch_bounds__(128, 2)
outer_mma_kernel(const unsigned char *__restrict__ aimg, const unsigned char *__restrict__ bimg, int rtiles, int ctiles,
                 int kch, const OuterShape S, float2 scale, float2 *__restrict__ out, int *err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char *sm = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  unsigned char *sa = sm, *sb = sm + 2 * kABlock;
  __shared__ __align__(8) uint64_t load_bar, mma_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int stop;
  __shared__ uint64_t col_at[kCols], row_at[kRows];  // x_A of a tile's columns, x_B of its rows
  const int tid = threadIdx.x, warp = tid >> 5, nA = S.nA;
  if (FIXED || SCALED) {
    col_at[tid] = FIXED ? spread(tid, S.a_bit, 7) : tid;
    row_at[tid] = FIXED ? spread(tid, S.b_bit, 7) : tid;
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&load_bar)));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&mma_bar)));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    stop = 0;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(smem_u32(&tmem_slot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  uint32_t lph = 0, mph = 0;  // parities of the two barriers
  bool load_out = false, mma_out = false;  // tid 0: a copy / products not yet waited for
  const uint64_t ntiles = (uint64_t)rtiles * ctiles;
  for (uint64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const uint64_t rt = tile / ctiles, ct = tile % ctiles;
    const uint64_t xa0 = FIXED ? spread(ct * kCols, S.a_bit, nA) : ct * kCols;
    const uint64_t xb0 = FIXED ? spread(rt * kRows, S.b_bit, S.nB) : rt * kRows;
    // the slices that the tile's fixed bits select
    uint64_t slice_a = 0, slice_b = 0;
    if (FIXED) {
      for (int j = 0; j < S.fix_a; ++j) slice_a |= ((xb0 >> S.fix_a_by[j]) & 1ull) << j;
      for (int j = 0; j < S.fix_b; ++j) slice_b |= ((xa0 >> S.fix_b_by[j]) & 1ull) << j;
    }
    for (int kc = 0; kc < kch; ++kc) {
      if (tid == 0) {
        const uint32_t lb = smem_u32(&load_bar);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(lb), "r"(kSmem) : "memory");
        const unsigned char *ga = aimg + ((slice_b * rtiles + rt) * kch + kc) * 2 * kABlock;
        const unsigned char *gb = bimg + ((slice_a * ctiles + ct) * kch + kc) * 2 * kBBlock;
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(smem_u32(sa)), "l"(ga), "r"(2 * kABlock), "r"(lb) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(smem_u32(sb)), "l"(gb), "r"(kBBlock), "r"(lb) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(smem_u32(sb + kBBlock)), "l"(gb + kBBlock), "r"(kBBlock), "r"(lb) : "memory");
        load_out = true;
        bool ok = mbar_wait(&load_bar, lph);
        if (ok) {
          load_out = false;
          lph ^= 1;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint64_t ah = sdesc(smem_u32(sa)), al = sdesc(smem_u32(sa + kABlock));
          const uint64_t bh = sdesc(smem_u32(sb)), bl = sdesc(smem_u32(sb + kBBlock));
          // one K step = 8 tf32 values = two 128-byte core matrices (+256 B = +16)
#pragma unroll
          for (int k = 0; k < kKc / 8; ++k) mma_ss(tmem, al + 16 * k, bh + 16 * k, kc > 0 || k > 0);
#pragma unroll
          for (int k = 0; k < kKc / 8; ++k) mma_ss(tmem, ah + 16 * k, bl + 16 * k, 1);
#pragma unroll
          for (int k = 0; k < kKc / 8; ++k) mma_ss(tmem, ah + 16 * k, bh + 16 * k, 1);
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                       ::"r"(smem_u32(&mma_bar)) : "memory");
          mma_out = true;
          ok = mbar_wait(&mma_bar, mph);
          if (ok) {
            mma_out = false;
            mph ^= 1;
          }
        }
        if (!ok) {
          atomicExch(err, 1);
          stop = 1;
        }
      }
      __syncthreads();
      if (stop) break;
    }
    if (stop) break;
    // D to the state: each warp holds 32 rows (x_B = rt * 128 + 32 warp + lane, one per
    // lane); per 32-column chunk the lanes write their rows into shared memory (the
    // operand buffers are free now: 4 KB per warp, 16-byte chunk q of row r at q ^ (r & 7),
    // conflict-free both ways), then the warp writes four rows' 128-byte runs per store
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t taddr = tmem + ((uint32_t)(32 * warp) << 16);
    const int lane = tid & 31;
    // the absorbed CZs' signs: the bits of x_A whose parity is this lane's row's sign
    uint64_t sign_mask = 0;
    if (SCALED)
      for (int j = 0; j < S.signs; ++j)
        sign_mask ^= (((xb0 + row_at[32 * warp + lane]) >> S.sign_b[j]) & 1ull) << S.sign_a[j];
    const uint32_t sign_base = __popcll(sign_mask & xa0);
    float4 *stg = reinterpret_cast<float4 *>(sa) + warp * 256;
    float2 *const rows = out + ((xb0 + (uint64_t)(32 * warp)) << nA) + xa0;
    const bool neighbours = !FIXED || S.a_bit[0] == 0;
    auto scaled = [&](uint32_t v) {
      const float x = __uint_as_float(v);
      return SCALED ? fmaf(x, scale.x, x * scale.y) : x * scale.x;
    };
#pragma unroll 1
    for (int c = 0; c < 256; c += 32) {
      uint32_t r[32];
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
          "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
            "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
            "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
            "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
          : "r"(taddr + (uint32_t)c)
          : "memory");
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (SCALED && sign_mask) {
#pragma unroll
        for (int q = 0; q < 32; ++q)  // (column c / 2 + q / 2 of the tile)
          r[q] ^= (sign_base + __popcll(sign_mask & col_at[c / 2 + q / 2])) << 31;
      }
#pragma unroll
      for (int q = 0; q < 8; ++q)
        stg[lane * 8 + (q ^ (lane & 7))] =
            make_float4(scaled(r[4 * q]), scaled(r[4 * q + 1]), scaled(r[4 * q + 2]), scaled(r[4 * q + 3]));
      __syncwarp();
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int row = 4 * q + (lane >> 3), ch = lane & 7;
        const float4 v = stg[row * 8 + (ch ^ (row & 7))];
        float2 *const to = FIXED ? out + ((xb0 + row_at[32 * warp + row]) << nA) + xa0 + col_at[c / 2 + 2 * ch]
                                 : rows + ((uint64_t)row << nA) + c / 2 + 2 * ch;
        if (neighbours) {
          *reinterpret_cast<float4 *>(to) = v;
        } else {
          to[0] = make_float2(v.x, v.y);
          to[1ull << S.a_bit[0]] = make_float2(v.z, v.w);
        }
      }
      __syncwarp();
    }
    // the next tile's products overwrite D only after every thread has read it, and its
    // bulk copies refill the staging buffer only after these generic-proxy writes
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
  }
  // after a wait that gave up: let the copy and the products in flight finish (bounded)
  // before the CTA's shared and tensor memory go away
  if (tid == 0 && load_out) mbar_wait(&load_bar, lph);
  if (tid == 0 && mma_out) mbar_wait(&mma_bar, mph);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem));
  }
}

}  // namespace

bool outer_sum_tc_supported(const OuterShape &S) { return S.a_free >= 7 && S.b_free >= 7 && S.t >= 0 && S.t <= 20; }

size_t outer_sum_tc_scratch(const OuterShape &S) {
  const uint64_t kch = ((2ull << S.t) + kKc - 1) / kKc;
  return (size_t)((((1ull << S.nB) << S.fix_b) / kRows) * kch * 2 * kABlock +
                  (((1ull << S.nA) << S.fix_a) / kCols) * kch * 2 * kBBlock);
}

cudaError_t launch_outer_sum_tc(const float2 *A, const float2 *B, const OuterShape &S, float2 scale, float2 *out,
                                void *scratch, int *err, cudaStream_t st) {
  if (!outer_sum_tc_supported(S)) return cudaErrorInvalidValue;
  const int form = S.fix_a + S.fix_b > 0 ? 2 : S.signs > 0 || scale.y != 0.f ? 1 : 0;
  const auto kernel = form == 0   ? outer_mma_kernel<false, false>
                      : form == 1 ? outer_mma_kernel<false, true>
                                  : outer_mma_kernel<true, true>;
  static bool configured[3] = {};
  if (!configured[form]) {
    const cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem + 1024);
    if (e != cudaSuccess) return e;
    configured[form] = true;
  }
  const int kch = (int)(((2ull << S.t) + kKc - 1) / kKc);
  const int rtiles = (int)((1ull << S.nB) / kRows), ctiles = (int)((1ull << S.nA) / kCols);
  unsigned char *aimg = static_cast<unsigned char *>(scratch);
  unsigned char *bimg = aimg + ((size_t)rtiles << S.fix_b) * kch * 2 * kABlock;
  const uint64_t work = (((1ull << S.nB) << S.fix_b) + ((2ull << S.nA) << S.fix_a)) * (uint64_t)kch * kKc;
  uint64_t pgrid = (work + 255) / 256;
  const uint64_t pmax = (uint64_t)device_sm_count() * 8;
  if (pgrid > pmax) pgrid = pmax;
  (form == 2 ? outer_prep_kernel<true> : outer_prep_kernel<false>)<<<(unsigned)pgrid, 256, 0, st>>>(A, B, S, kch, aimg, bimg);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  uint64_t grid = (uint64_t)device_sm_count() * 2;
  const uint64_t ntiles = (uint64_t)rtiles * ctiles;
  if (grid > ntiles) grid = ntiles;
  kernel<<<(unsigned)grid, 128, kSmem + 1024, st>>>(aimg, bimg, rtiles, ctiles, kch, S, scale, out, err);
  return cudaGetLastError();
}

}  // namespace svk
