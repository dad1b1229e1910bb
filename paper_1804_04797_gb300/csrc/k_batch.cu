// K7: the uneven batch in one persistent launch.
//
// Every CTA repeatedly takes the next item (a run of tiles of one pass of one circuit) from a
// global counter and runs the plain tile pass on them.  Before an item of pass p it waits
// until every tile of pass p-1 of the same circuit is done (a per-circuit-pass counter),
// with a bounded spin: a wait that gives up sets the error word and the CTA leaves.  The
// queue holds all circuits' first passes, then all second passes, ..., so the waits are
// rare and short.  The state is read through L2 only (cp.async.cg), because other CTAs
// of the same launch wrote it and L1 is not coherent across SMs.  The tile pass is the
// interpreter of the single-circuit path (tile_interp.cuh).
#include <cuda_runtime.h>

#include "batch.h"
#include "kernels.h"
#include "tile_interp.cuh"

namespace svk {
namespace {

using namespace itp;

constexpr int kBatchSlots = 4;  // register slots besides the pack bit

__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ unsigned int load_acquire(const unsigned int *p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__global__ void __launch_bounds__(256, 2)
batch_kernel(float2 *__restrict__ states, const unsigned char *__restrict__ blocks, const BatchCP *__restrict__ cps,
             const BatchItem *__restrict__ items, uint32_t n_items, unsigned int *words, uint32_t tile_bytes,
             unsigned long long wait_ns) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float4 *tile = reinterpret_cast<float4 *>(smem_raw);
  unsigned char *blk = smem_raw + tile_bytes;
  __shared__ unsigned int s_item;
  __shared__ int s_stop;
  const int tid = threadIdx.x;
  unsigned int *done = words + kBatchHeader;
  uint32_t cur_cp = kNoPrev;
  for (;;) {
    if (tid == 0) {
      s_item = atomicAdd(&words[0], 1u);
      s_stop = 0;
    }
    __syncthreads();
    const unsigned int idx = s_item;
    if (idx >= n_items) break;
    const BatchItem it = items[idx];
    const BatchCP cp = cps[it.cp];
    const unsigned char *src = blocks + cp.block;
    if (it.cp != cur_cp) {
      fetch_block(blk, src, cp.block_bytes);
      cur_cp = it.cp;
      if (tid == 0 && cp.prev != kNoPrev) {
        const unsigned int need = cps[cp.prev].tiles;
        if (load_acquire(&done[cp.prev]) < need) {
          const unsigned long long t0 = now_ns();
          while (load_acquire(&done[cp.prev]) < need) {
            if (now_ns() - t0 > wait_ns) {
              atomicExch(&words[1], 1u);
              s_stop = 1;
              break;
            }
          }
        }
      }
    }
    __syncthreads();
    if (s_stop) break;
    const uint32_t end = min(it.tile + (1u << cp.run), cp.tiles);
    for (uint32_t t = it.tile; t < end; ++t) process_tile<kBatchSlots>(states + cp.state_off, blk, src, tile, t);
    __threadfence();  // each thread's stores visible device-wide before the count
    __syncthreads();
    if (tid == 0) atomicAdd(&done[it.cp], end - it.tile);
  }
}

__global__ void pick_kernel(const float2 *__restrict__ psi, const __grid_constant__ PickArgs args, int count,
                            float2 *__restrict__ out) {
  const int i = threadIdx.x;
  if (i < count) out[i] = psi[args.index[i]];
}

// The queue, written where it is read: built by the host it took 0.48 ms of a call on 64 new
// circuits of 10..22 qubits (137 k items, one push each, and their copy).
__global__ void items_kernel(const BatchCP *__restrict__ cps, uint32_t n_cps, BatchItem *__restrict__ items,
                             uint32_t n_items) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_items) return;
  uint32_t at = 0, end = n_cps;  // the last circuit-pass that starts at or before the item
  while (end - at > 1) {
    const uint32_t mid = at + (end - at) / 2;
    if (cps[mid].first <= i) at = mid;
    else end = mid;
  }
  items[i] = BatchItem{at, (i - cps[at].first) << cps[at].run};
}

__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

__global__ void batch_stats_partial(const float2 *__restrict__ states, const BatchChunk *__restrict__ chunks,
                                    double *partials) {
  const BatchChunk ch = chunks[blockIdx.x];
  // two amplitudes per 16-byte load: chunk starts and lengths are even (every circuit
  // has at least 2^6 amplitudes, chunks are 2^16); eight probabilities are added in
  // fp32, then into the fp64 sums (fp64 per element is the slow part on this GPU)
  const float4 *p = reinterpret_cast<const float4 *>(states + ch.start);
  const uint32_t n4 = ch.len >> 1, stride = blockDim.x;
  double s2 = 0, s4 = 0;
  uint32_t i = threadIdx.x;
  for (; i + 3 * stride < n4; i += 4 * stride) {
    float4 z[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) z[k] = p[i + k * stride];
    float a2 = 0.f, a4 = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float p0 = fmaf(z[k].x, z[k].x, z[k].y * z[k].y);
      const float p1 = fmaf(z[k].z, z[k].z, z[k].w * z[k].w);
      a2 += p0 + p1;
      a4 = fmaf(p0, p0, fmaf(p1, p1, a4));
    }
    s2 += a2;
    s4 += a4;
  }
  for (; i < n4; i += stride) {
    const float4 z = p[i];
    const float p0 = fmaf(z.x, z.x, z.y * z.y);
    const float p1 = fmaf(z.z, z.z, z.w * z.w);
    s2 += (double)(p0 + p1);
    s4 += (double)fmaf(p0, p0, p1 * p1);
  }
  __shared__ double r2[8], r4[8];
  s2 = warp_sum(s2);
  s4 = warp_sum(s4);
  if ((threadIdx.x & 31) == 0) { r2[threadIdx.x >> 5] = s2; r4[threadIdx.x >> 5] = s4; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = 0, b = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) { a += r2[w]; b += r4[w]; }
    partials[2 * blockIdx.x] = a;
    partials[2 * blockIdx.x + 1] = b;
  }
}

__global__ void batch_stats_final(const double *partials, const int *chunk_begin, int n_circuits, double *stats) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n_circuits) return;
  double a = 0, b = 0;
  for (int k = chunk_begin[c]; k < chunk_begin[c + 1]; ++k) { a += partials[2 * k]; b += partials[2 * k + 1]; }
  stats[2 * c] = a;
  stats[2 * c + 1] = b;
}

}  // namespace

int batch_block_threads(int m) { return 1 << (m - 1 - kBatchSlots); }

namespace {
size_t batch_smem(uint32_t max_block_bytes, int m) {
  return (sizeof(float2) << m) + svp::interp_smem_max(max_block_bytes) + svp::kInterpPad;
}
}  // namespace

// An item's fixed cost -- the counter, the item, the pass's program, the dependency, the fence
// and the count -- is shared by its tiles, but a pass ends with the last of its items, so the
// runs grow with the tiles that every CTA has to take (us at runs of 1 / 2 / 4 / 8 / 16 tiles):
//   40 circuits of 8..10 qubits 61 / 77 / 111 / 109 / 109, 84 of 11..18 190 / 224 / 353 / 520 / 757,
//   512 of 12..16 403 / 411 / 450 / 570 / 860, 64 of 10..22 1265 / 1249 / 1304 / 1445 / 2002,
//   96 of 14..22 1913 / 1834 / 1810 / 1805 / 1920, 256 of 16..23 12837 / 12362 / 12167 / 12083 / 12055.
// A small circuit's pass keeps 64 items.
int batch_run_log(uint32_t tiles, double per_cta) {
  int run = 0;
  while (run < 4 && per_cta >= 16 << run && tiles >= 128u << run) ++run;
  return run;
}

int batch_grid(uint32_t max_block_bytes, int m) {
  static bool configured = false;
  if (!configured) {  // tiles of <= 13 qubits (capi_batch)
    if (cudaFuncSetAttribute(batch_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)batch_smem(svp::kInterpResident, 13)) != cudaSuccess)
      return 0;
    configured = true;
  }
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, batch_kernel, batch_block_threads(m),
                                                    batch_smem(max_block_bytes, m)) != cudaSuccess)
    return 0;
  return device_sm_count() * (per_sm < 1 ? 1 : per_sm);
}

cudaError_t launch_batch(float2 *states, const unsigned char *blocks, uint32_t max_block_bytes, const BatchCP *cps,
                         const BatchItem *items, uint32_t n_items, unsigned int *words, int m, cudaStream_t st,
                         unsigned long long wait_ns, int max_grid) {
  int grid = batch_grid(max_block_bytes, m);
  if (grid < 1) return cudaGetLastError();
  if (max_grid > 0 && grid > max_grid) grid = max_grid;
  batch_kernel<<<grid, batch_block_threads(m), batch_smem(max_block_bytes, m), st>>>(
      states, blocks, cps, items, n_items, words, (uint32_t)(sizeof(float2) << m), wait_ns);
  return cudaGetLastError();
}

cudaError_t launch_pick(const float2 *psi, const PickArgs &args, int count, float2 *out, cudaStream_t st) {
  if (count < 1 || count > kPickMost) return cudaErrorInvalidValue;
  pick_kernel<<<1, (count + 31) / 32 * 32, 0, st>>>(psi, args, count, out);
  return cudaGetLastError();
}

cudaError_t launch_batch_items(const BatchCP *cps, uint32_t n_cps, BatchItem *items, uint32_t n_items,
                               cudaStream_t st) {
  items_kernel<<<(n_items + 255) / 256, 256, 0, st>>>(cps, n_cps, items, n_items);
  return cudaGetLastError();
}

cudaError_t launch_batch_stats(const float2 *states, const BatchChunk *chunks, int n_chunks, double *partials,
                               const int *chunk_begin, int n_circuits, double *stats, cudaStream_t st) {
  if (n_chunks > 0) batch_stats_partial<<<n_chunks, 256, 0, st>>>(states, chunks, partials);
  batch_stats_final<<<(n_circuits + 127) / 128, 128, 0, st>>>(partials, chunk_begin, n_circuits, stats);
  return cudaGetLastError();
}

}  // namespace svk
