// Work queue of the uneven batch (one persistent launch over many circuits).
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.h"

namespace svk {

// One pass of one circuit.  Its tiles are items of 2^run neighbouring ones (up to the last);
// `first` is its first item.
struct BatchCP {
  uint64_t state_off;  // float2 offset of the circuit's state in the batch buffer
  uint64_t block;      // offset of the pass's block (interp_dev.h) in the batch program
  uint32_t block_bytes;
  uint32_t prev;       // BatchCP index of the circuit's previous pass (kNoPrev if first)
  uint32_t tiles;      // tiles of this pass
  uint32_t first;
  uint32_t run;
};
constexpr uint32_t kNoPrev = 0xFFFFFFFFu;

// The tiles from `tile` on, of one circuit-pass.  Items are dispensed in array order: all first
// passes, then all second passes, ...; an item waits only for its circuit's previous pass, which
// was dispensed earlier to a CTA that is already running, so the queue cannot deadlock.
struct BatchItem {
  uint32_t cp;
  uint32_t tile;
};
// The queue, from its circuit-passes (in order of `first`).
cudaError_t launch_batch_items(const BatchCP *cps, uint32_t n_cps, BatchItem *items, uint32_t n_items, cudaStream_t st);

// Device words of one launch: [0] next item, [1] error flag, then one done counter per cp.
constexpr int kBatchHeader = 2;

// The run of a pass of `tiles` tiles (BatchCP::run), in a batch whose passes have `per_cta` tiles
// for each of the launch's CTAs on average.
int batch_run_log(uint32_t tiles, double per_cta);
// CTAs of a launch (max_block_bytes: the largest of the programs).
int batch_grid(uint32_t max_block_bytes, int m);

// blocks: the circuit-passes' programs.  wait_ns: limit of one dependency wait (after which the
// error word is set and the CTA leaves); max_grid > 0 caps the number of CTAs.
cudaError_t launch_batch(float2 *states, const unsigned char *blocks, uint32_t max_block_bytes, const BatchCP *cps,
                         const BatchItem *items, uint32_t n_items, unsigned int *words, int m, cudaStream_t st,
                         unsigned long long wait_ns = 5000000000ull, int max_grid = 0);
int batch_block_threads(int m);

// out[i] = psi[index[i]], i < count: the indices ride in the launch's arguments.
constexpr int kPickMost = 256;
struct PickArgs {
  uint64_t index[kPickMost];
};
cudaError_t launch_pick(const float2 *psi, const PickArgs &args, int count, float2 *out, cudaStream_t st);

// Per-circuit fp64 norm and sum |alpha|^4: chunk c covers [start, start + len) of circuit
// circ; partials (2 doubles per chunk) then one thread per circuit adds its chunks in order.
struct BatchChunk {
  uint64_t start;
  uint32_t len;
  uint32_t circuit;
};
cudaError_t launch_batch_stats(const float2 *states, const BatchChunk *chunks, int n_chunks, double *partials,
                               const int *chunk_begin, int n_circuits, double *stats, cudaStream_t st);

}  // namespace svk
