// Program of one tile pass as the interpreting kernels read it: the pass's header, its
// stages, steps and gates in one contiguous block, so that a CTA fetches it into shared memory
// with one round of coalesced 16-byte loads (the kernels' former reads of pass, stage,
// group-table and op records from global memory, each dependent on the one before, were
// their first stall: 2-4 cycles per issued instruction on states of 12 to 20 qubits).
#pragma once

#include <cstdint>

#include "plan_dev.h"

namespace svp {

// A thread's slots: register slots 0..3 and 4 = the pack bit.
constexpr int kInterpPack = 4;
constexpr int kInterpMaxSlots = 4;  // register slots besides the pack bit

// Gates on the register bits (codes + slot; interp_gates.cuh runs them).  The signs of a
// slot's 1 elements (Z, and CZ with a qubit fixed for the thread) collect into one parity
// over the thread's condition word W, its top bit set: -1 where popc(W & par) is odd.
enum GCode : uint32_t {
  // the square roots as unscaled rotations after the slot's sign; s = 1, or -1 for the
  // adjoint (kGateAdj)
  G_IM = 0,    // X^{1/2}: x' = x - i s y, y' = y - i s x
  G_RE = 5,    // Y^{1/2}: x' = x - s y, y' = y + s x
  G_H = 10,    // x' = x + y, y' = x - y (its factor 1/sqrt2 is a G_RS)
  G_T = 15,    // slot-1 elements times (1 + i s) c, c a rounding of 1/sqrt2: the lower one, or
               // the upper one (kGateUp)
  G_SIGN = 20, // the slot's sign alone
  G_CZ = 25,   // + pair of slots: -1 where both are 1
  G_RS = 35,   // every element times 1/sqrt2
  G_END = 36
};
constexpr uint32_t kGateAdj = 0x80000000u, kGateUp = 0x40000000u, kParityOne = 0x80000000u;
struct IGate {
  uint32_t w, par;  // code and flags; the parity mask
};

// Steps of a pass.  Conditions: (W & wmask) == wval.
enum ICode : uint32_t {
  I_RUN = 0,    // the gates from index arg on (wmask of them, an even number, with the G_END)
  I_PHASE,      // the thread's scalar phase += arg where the condition holds (arg 0: its
                // elements are to be zeroed)
  I_MASKMUL,    // elements under the mask arg times 0 where the condition holds (projectors)
  I_MASKSET,    // the same set to 0 (branch projectors)
  I_SCALAR,     // every element times arg (a power of two) and e^{i pi q/4} 2^{-u/2}, q = wmask and
                // u = wval; q = kStageEnd: the phase and the zeroing recorded in the stage
  // moves (arg of I_LOAD and I_STORE: the stage)
  I_INIT,       // the initial state into registers
  I_IN,         // global memory -> registers (the first stage's lanes cover contiguous runs)
  I_FETCH,      // global memory -> tile
  I_LOAD,       // tile -> registers; wval = 1: after I_FETCH
  I_STORE,      // registers -> tile
  I_OUT,        // registers -> global memory
  I_SWEEP,      // tile -> global memory
  I_COUNT
};
constexpr uint32_t kStageEnd = 8;
// Element masks: bit p (+ 16 for the pack bit's 1) of pair p.

struct IStep {
  uint32_t code, arg, wmask, wval;
};
static_assert(sizeof(IStep) == 16 && sizeof(IGate) == 8, "step layout");

struct IStage {
  uint32_t reg[4];  // shared-memory byte-offset masks of the register slots
  uint32_t L[48];   // group addressing: see DevGroupEntry (byte offsets)
};
static_assert(sizeof(IStage) == 208, "IStage layout");

// A run of consecutive qubits outside the tile: ((tile_id >> from) & mask) << to.
struct IRun {
  uint32_t mask;
  uint8_t from, to;
  uint16_t pad;
};

struct IHead {
  uint32_t bytes;                 // of the whole block (a multiple of 16)
  uint32_t stage_count, step_count, gate_count;
  uint8_t m, runs, flags, pad;    // flags: PassFlags
  float init_amp;
  uint32_t pad2[2];
  uint8_t tq[16];
  IRun run[12];
  uint64_t it_off[16];            // global offset of pair index i << (m - 1 - register slots)
  // global offsets of the group bits (0..11) and register slots (12..15) of the first and
  // the last stage
  uint64_t gin[16], gout[16];
};
static_assert(sizeof(IHead) % 16 == 0, "IHead layout");

// What a CTA holds of a block at once: all of it where it is small enough, else the header
// and one run of gates.
constexpr uint32_t kInterpRun = 512;  // gates of a run, with its end
constexpr uint32_t kInterpResident = 12288;  // bytes
constexpr uint32_t interp_smem_bytes(uint32_t block) {
  return block <= kInterpResident ? block : (uint32_t)(sizeof(IHead) + kInterpRun * sizeof(IGate));
}
// (the entry after a run's end is read, never used)
constexpr uint32_t kInterpPad = 16;
// The most a block of at most `block` bytes takes.
constexpr uint32_t interp_smem_max(uint32_t block) {
  return block <= interp_smem_bytes(kInterpResident + 1) ? interp_smem_bytes(kInterpResident + 1)
         : block <= kInterpResident                      ? block
                                                         : kInterpResident;
}

}  // namespace svp
