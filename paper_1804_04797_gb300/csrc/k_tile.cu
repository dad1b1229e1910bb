// Plain (fp32 CUDA-core) tile pass, interpreting the plan.
//
// One launch = one pass of the plan = one read and one write of every amplitude.
// Each CTA loops over gathered tiles: the 2^m amplitudes whose indices differ only in
// the pass's m tile qubits (the c lowest qubits are always among them, so the tile is
// 2^(m-c) contiguous chunks of 2^c amplitudes and every global access is a coalesced
// 16-byte vector).  The tile is staged in shared memory (the on-chip copy of the
// paper's "local qubits" in LDM, §2.3) and every gate of the pass is applied to it:
// stage by stage, each thread pulls the amplitudes that differ in the stage's qubits
// (qubit 0, the pack bit, and two or four register qubits) into registers as packed pairs,
// applies the stage's gates there (the pair update of §2 with packed fp32x2 arithmetic;
// diagonal gates as signs, phases and projector factors, conditioned on the thread's other
// index bits), and writes them back (tile_interp.cuh).  Tile size and register width by
// state size: interp_shape in capi.cpp.
#include <cuda_runtime.h>

#include <algorithm>

#include "kernels.h"
#include "tile_interp.cuh"

namespace svk {
namespace {

using namespace itp;

constexpr int kMaxBits = 13;  // tiles of this kernel: 64 KiB

// RK: register slots besides the pack bit (2^(RK + 1) amplitudes a thread).
template <int RK>
__global__ void __launch_bounds__(1 << (kMaxBits - 1 - RK), RK == 2 ? 1 : 2)
tile_pass_kernel(float2 *__restrict__ psi, const unsigned char *__restrict__ block, uint32_t bytes, uint32_t tile_bytes,
                 uint64_t num_tiles) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned char *blk = smem_raw + tile_bytes;
  fetch_block(blk, block, bytes);
  __syncthreads();
  for (uint64_t tile_id = blockIdx.x; tile_id < num_tiles; tile_id += gridDim.x)
    process_tile<RK>(psi, blk, block, reinterpret_cast<float4 *>(smem_raw), tile_id);
}

template <int RK>
cudaError_t launch(float2 *psi, int n, const unsigned char *block, uint32_t bytes, int m, cudaStream_t st) {
  const size_t tile_bytes = sizeof(float2) << m, smem = tile_bytes + svp::interp_smem_bytes(bytes) + svp::kInterpPad;
  static bool configured = false;
  if (!configured) {
    cudaError_t e = cudaFuncSetAttribute(
        tile_pass_kernel<RK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
        (int)((sizeof(float2) << kMaxBits) + svp::kInterpResident + svp::kInterpPad));
    if (e != cudaSuccess) return e;
    configured = true;
  }
  const int threads = 1 << (m - 1 - RK);
  const uint64_t tiles = 1ull << (n - m);
  uint64_t grid = tiles;
  if (grid > (uint64_t)device_sm_count()) {
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, tile_pass_kernel<RK>, threads, smem);
    if (e != cudaSuccess) return e;
    grid = std::min(grid, (uint64_t)device_sm_count() * (uint64_t)(per_sm < 1 ? 1 : per_sm));
  }
  tile_pass_kernel<RK><<<(unsigned)grid, threads, smem, st>>>(psi, block, bytes, (uint32_t)tile_bytes, tiles);
  return cudaGetLastError();
}

}  // namespace

int tile_pass_max_bits() { return kMaxBits; }

cudaError_t launch_tile_pass(float2 *psi, int n, const unsigned char *block, uint32_t bytes, int m, int rk,
                             cudaStream_t st) {
  if (m < rk + 2 || m > kMaxBits || m > n) return cudaErrorInvalidValue;
  switch (rk) {
    case 2: return launch<2>(psi, n, block, bytes, m, st);
    case 4: return launch<4>(psi, n, block, bytes, m, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace svk
