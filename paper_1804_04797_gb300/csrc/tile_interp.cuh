// Interpreter of packed plans: the tile pass of states below the size from which plans are
// compiled, of batches, and wherever there is no run-time compiler.
//
// A thread holds 2^RK pairs of amplitudes and runs a stage's gates on them in registers
// (interp_gates.cuh).  What bounds these kernels is not arithmetic but everything around it:
// the pass's program is one block that a CTA fetches into shared memory at once (the
// dependent reads of pass, stage and op records were the first stall of small states),
// signs of a slot are collected into one parity, and where a stage's lanes cover contiguous
// runs of global memory its registers are loaded from, or stored to, global memory directly
// (no asynchronous copy, regrouping sweep and barrier).
//
// The values are those of the plan kernels without pipelining (jit.cpp, pass_source), bit
// for bit.
#pragma once

#include "interp_gates.cuh"

namespace svk {
namespace itp {

using svp::IHead;
using svp::IStage;
using svp::IStep;

constexpr float kS2 = 0.70710678118654752440f;
constexpr float kS2lo = 1.21016171e-8f;  // 1/sqrt2 - kS2: v*kS2 + v*kS2lo rounds v/sqrt2 to nearest

// ---- packed values ---------------------------------------------------------------------------

__device__ __forceinline__ P2 pk(float a, float b) {
  P2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 un(P2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ P2 pfma(P2 a, P2 b, P2 c) {
  P2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ P2 pmul(P2 a, P2 b) {
  P2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// v/sqrt2, the factor as hi + lo
__device__ __forceinline__ P2 prs(P2 v) { return pfma(v, pk(kS2, kS2), pmul(v, pk(kS2lo, kS2lo))); }

// ---- scalars and masks ----------------------------------------------------------------------

template <int RK>
__device__ __forceinline__ void scale(PRegs<RK> &R, PRegs<RK> &I, float f) {
  const P2 ff = pk(f, f);
#pragma unroll
  for (int p = 0; p < (1 << RK); ++p) {
    R[p] = pmul(R[p], ff);
    I[p] = pmul(I[p], ff);
  }
}
// every element times 1/sqrt2
template <int RK>
__device__ __forceinline__ void rs_all(PRegs<RK> &R, PRegs<RK> &I) {
#pragma unroll
  for (int p = 0; p < (1 << RK); ++p) {
    R[p] = prs(R[p]);
    I[p] = prs(I[p]);
  }
}
// Every element times e^{i pi q/4} 2^{-u/2}: (c + i d)/sqrt2 for odd q, so that u = 1 leaves
// an exact 1/2 (the forms of phase_all and global_factor).
template <int RK>
__device__ __forceinline__ void phase_scalar(PRegs<RK> &R, PRegs<RK> &I, uint32_t q, uint32_t u) {
  if (q & 1) {
    const float c = (q == 1 || q == 7) ? 1.f : -1.f, d = (q == 1 || q == 3) ? 1.f : -1.f;
    const P2 c2 = pk(c, c), d2 = pk(d, d), m2 = pk(-d, -d);
#pragma unroll
    for (int p = 0; p < (1 << RK); ++p) {
      const P2 r = pfma(I[p], m2, pmul(R[p], c2));
      I[p] = pfma(I[p], c2, pmul(R[p], d2));
      R[p] = r;
    }
  } else if (q) {
    // times i^{q/2}: q = 2 (-i, r), 4 (-r, -i), 6 (i, -r)
    const float a = q == 6 ? 1.f : -1.f, b = q == 2 ? 1.f : -1.f;
    const bool swap = q != 4;
    const P2 a2 = pk(a, a), b2 = pk(b, b);
#pragma unroll
    for (int p = 0; p < (1 << RK); ++p) {
      const P2 r = R[p];
      R[p] = pmul(swap ? I[p] : r, a2);
      I[p] = pmul(swap ? r : I[p], b2);
    }
  }
  u += q & 1;
  if (u == 2) scale<RK>(R, I, 0.5f);
  if (u == 1) rs_all<RK>(R, I);
}
// Elements under `mask` set to zero (set) or multiplied by 0 (the sign of zero of the
// plan kernels' projector factors).
template <int RK>
__device__ __forceinline__ void mask_zero(PRegs<RK> &R, PRegs<RK> &I, uint32_t mask, bool set) {
#pragma unroll
  for (int p = 0; p < (1 << RK); ++p) {
    const bool x = (mask >> p) & 1u, y = (mask >> (p + 16)) & 1u;
    const P2 f = pk(x ? 0.f : 1.f, y ? 0.f : 1.f);
    float2 r = un(pmul(R[p], f)), i = un(pmul(I[p], f));
    if (set && x) r.x = i.x = 0.f;
    if (set && y) r.y = i.y = 0.f;
    R[p] = pk(r.x, r.y);
    I[p] = pk(i.x, i.y);
  }
}

// ---- a pass's program -------------------------------------------------------------------------

// 16 bytes per thread and turn.
__device__ __forceinline__ void copy16(unsigned char *dst, const unsigned char *src, uint32_t bytes) {
  for (uint32_t i = threadIdx.x; i < bytes / 16; i += blockDim.x)
    reinterpret_cast<uint4 *>(dst)[i] = __ldg(reinterpret_cast<const uint4 *>(src) + i);
}
// A pass's block into shared memory (its header only where it is too large to stay there).
__device__ __forceinline__ void fetch_block(unsigned char *blk, const unsigned char *src, uint32_t bytes) {
  copy16(blk, src, bytes <= svp::kInterpResident ? bytes : (uint32_t)sizeof(IHead));
}

// Global offset of thread t's group in the first or last stage (g: IHead's gin or gout).
__device__ __forceinline__ uint64_t group_offset(const uint64_t *g, uint32_t t, int bits) {
  uint64_t o = 0;
  for (int i = 0; i < bits; ++i)
    if ((t >> i) & 1u) o += g[i];
  return o;
}
// Byte offset of pair p of a thread's group in the tile (a0: of its first pair).
__device__ __forceinline__ uint32_t slot_offset(uint32_t a0, const uint4 &reg, int p) {
  if (p & 1) a0 ^= reg.x;
  if (p & 2) a0 ^= reg.y;
  if (p & 4) a0 ^= reg.z;
  if (p & 8) a0 ^= reg.w;
  return a0;
}
// 16-byte slot of pair k (plan.h, pack_phys, layout 0).
__device__ __forceinline__ uint32_t pair_slot(uint32_t k) { return k ^ (((k >> 3) ^ (k >> 6) ^ (k >> 9)) & 7u); }
__device__ __forceinline__ uint32_t group_slot(const IStage &st, uint32_t t) {
  return st.L[t & 15] ^ st.L[16 + ((t >> 4) & 15)] ^ st.L[32 + (t >> 8)];
}

// One tile of a pass: its program from the read (or the initial state) to the write.  blk:
// the pass's block as fetch_block left it, src: the block in global memory.  One loop runs
// every step, the moves between memory and registers among them, so that each one's code
// exists once.  Ends with __syncthreads.
template <int RK>
__device__ __forceinline__ void process_tile(float2 *__restrict__ psi, unsigned char *blk, const unsigned char *src,
                                             float4 *tile, uint64_t tile_id) {
  using namespace svp;
  const IHead &H = *reinterpret_cast<const IHead *>(blk);
  const uint32_t tid = threadIdx.x, T = blockDim.x;
  const bool resident = H.bytes <= kInterpResident;
  const int bits = H.m - 1 - RK;
  float2 *at = psi;
  for (int i = 0; i < H.runs; ++i) at += ((tile_id >> H.run[i].from) & (uint64_t)H.run[i].mask) << H.run[i].to;
  // condition word: the group index below the tile index (at most 32 bits)
  const uint32_t W = ((uint32_t)tile_id << bits) | tid;
  const uint32_t n_steps = H.step_count, steps_at = (uint32_t)sizeof(IHead) + H.stage_count * (uint32_t)sizeof(IStage);
  const uint32_t gates_at = steps_at + n_steps * (uint32_t)sizeof(IStep);
  const IStage *const stages = reinterpret_cast<const IStage *>((resident ? blk : src) + sizeof(IHead));
  const uint4 *const steps = reinterpret_cast<const uint4 *>((resident ? blk : src) + steps_at);
  const uint32_t gates = (uint32_t)__cvta_generic_to_shared(blk + (resident ? gates_at : (uint32_t)sizeof(IHead)));
  constexpr int kP = 1 << RK;
  PRegs<RK> R, I;
#pragma unroll
  for (int p = 0; p < kP; ++p) R[p] = I[p] = 0;
  int ph = 0;         // scalar phase, in eighths of a turn
  bool zero = false;  // the thread's elements are to be zeroed
#pragma unroll 1
  for (uint32_t o = 0; o < n_steps; ++o) {
    const uint4 h = steps[o];  // code, arg, wmask, wval
    switch (h.x) {
      case I_RUN:
        if (!resident) {
          __syncthreads();
          copy16(blk + sizeof(IHead), src + gates_at + (size_t)h.y * sizeof(IGate), h.z * (uint32_t)sizeof(IGate));
          __syncthreads();
        }
        run_gates<RK>(R, I, gates + (resident ? h.y * (uint32_t)sizeof(IGate) : 0u), W | kParityOne);
        break;
      case I_PHASE:
        if ((W & h.z) == h.w) {
          if (h.y) ph += (int)h.y;
          else zero = true;
        }
        break;
      case I_MASKMUL:
      case I_MASKSET: mask_zero<RK>(R, I, (W & h.z) == h.w ? h.y : 0u, h.x == I_MASKSET); break;
      case I_SCALAR: {  // scalars: a factor 2^-k, then a phase (one copy of their code)
        uint32_t q = h.z, u = h.w;
        float f = __uint_as_float(h.y);
        if (q == kStageEnd) {
          q = zero ? 0u : (uint32_t)ph & 7u;
          u = 0;
          if (zero) f = 0.f;
          ph = 0;
          zero = false;
        }
        if (f != 1.f) scale<RK>(R, I, f);
        if (q | u) phase_scalar<RK>(R, I, q, u);
        break;
      }
      case I_INIT: {
        const P2 v = (H.flags & PF_INIT_UNIFORM) ? pk(H.init_amp, H.init_amp) : 0;
#pragma unroll
        for (int p = 0; p < kP; ++p) { R[p] = v; I[p] = 0; }
        if (!(H.flags & PF_INIT_UNIFORM) && W == 0) R[0] = pk(1.f, 0.f);
        break;
      }
      case I_IN: {  // global memory -> registers
        const float2 *const from = at + group_offset(H.gin, tid, bits);
#pragma unroll
        for (int p = 0; p < kP; ++p) {
          uint64_t off = 0;
#pragma unroll
          for (int j = 0; j < RK; ++j)
            if ((p >> j) & 1) off += H.gin[12 + j];
          const float4 x = __ldcg(reinterpret_cast<const float4 *>(from + off));  // (re, im, re', im')
          R[p] = pk(x.x, x.z);
          I[p] = pk(x.y, x.w);
        }
        break;
      }
      case I_FETCH: {  // global memory -> tile, in the order of the state's pairs
        const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(tile);
        const float2 *from = at;
        for (int i = 0; i < bits; ++i)
          if ((tid >> i) & 1u) from += 1ull << H.tq[i + 1];
#pragma unroll 4
        for (int it = 0; it < kP; ++it)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sbase + 16u * pair_slot(tid + (uint32_t)it * T)),
                       "l"(from + H.it_off[it])
                       : "memory");
        asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
        __syncthreads();
        break;
      }
      case I_LOAD: {  // tile -> registers (cond word wval = 1: pairs as I_FETCH left them)
        const IStage &st = stages[h.y];
        const uint4 reg = *reinterpret_cast<const uint4 *>(st.reg);
        const uint32_t a0 = group_slot(st, tid);
        const bool copied = h.w != 0u;
#pragma unroll
        for (int p = 0; p < kP; ++p) {
          const float4 x = *reinterpret_cast<const float4 *>(reinterpret_cast<const char *>(tile) + slot_offset(a0, reg, p));
          R[p] = pk(x.x, copied ? x.z : x.y);
          I[p] = pk(copied ? x.y : x.z, x.w);
        }
        break;
      }
      case I_STORE: {  // registers -> tile
        const IStage &st = stages[h.y];
        const uint4 reg = *reinterpret_cast<const uint4 *>(st.reg);
        const uint32_t a0 = group_slot(st, tid);
#pragma unroll
        for (int p = 0; p < kP; ++p) {
          const float2 r = un(R[p]), i = un(I[p]);
          *reinterpret_cast<float4 *>(reinterpret_cast<char *>(tile) + slot_offset(a0, reg, p)) =
              make_float4(r.x, r.y, i.x, i.y);
        }
        __syncthreads();
        break;
      }
      case I_OUT: {  // registers -> global memory
        float2 *const to = at + group_offset(H.gout, tid, bits);
#pragma unroll
        for (int p = 0; p < kP; ++p) {
          uint64_t off = 0;
#pragma unroll
          for (int j = 0; j < RK; ++j)
            if ((p >> j) & 1) off += H.gout[12 + j];
          const float2 r = un(R[p]), i = un(I[p]);
          *reinterpret_cast<float4 *>(to + off) = make_float4(r.x, i.x, r.y, i.y);
        }
        break;
      }
      case I_SWEEP: {  // tile -> global memory, in the order of the state's pairs
        float2 *to = at;
        for (int i = 0; i < bits; ++i)
          if ((tid >> i) & 1u) to += 1ull << H.tq[i + 1];
#pragma unroll 4
        for (int it = 0; it < kP; ++it) {
          const float4 x = tile[pair_slot(tid + (uint32_t)it * T)];
          *reinterpret_cast<float4 *>(to + H.it_off[it]) = make_float4(x.x, x.z, x.y, x.w);
        }
        break;
      }
      default: break;
    }
  }
  __syncthreads();
}

}  // namespace itp
}  // namespace svk
