// Lowering of packed plans to the interpreting kernels' programs (interp_dev.h).
#include "interp.h"

#include <algorithm>
#include <cmath>
#include <cstring>

namespace svp {

namespace {

uint32_t bits_of(float f) {
  uint32_t u;
  std::memcpy(&u, &f, sizeof(u));
  return u;
}

// Elements of a thread (bit p, + 16 where the pack bit is 1) whose slot is 1.
uint32_t slot_mask(int slot) {
  if (slot == kInterpPack) return 0xffff0000u;
  uint32_t m = 0;
  for (int p = 0; p < 16; ++p)
    if ((p >> slot) & 1) m |= 0x10001u << p;
  return m;
}

int slot_of(int j) { return j == kPackSlot ? kInterpPack : j; }

// Index of a slot pair (j < k) after G_CZ: (0,1) (0,2) (0,3) (1,2) (1,3) (2,3) then (j, pack).
uint32_t cz_pair(int j, int k) {
  if (k == kInterpPack) return 6 + (uint32_t)j;
  return (uint32_t)(j == 0 ? k - 1 : j + k);
}

struct Lowering {
  std::vector<IStep> steps;
  std::vector<IGate> gates;
  bool open = false;  // the last step is a run that takes more gates

  void step(uint32_t code, uint32_t arg, uint32_t wmask, uint32_t wval) {
    close();
    steps.push_back(IStep{code, arg, wmask, wval});
  }
  void gate(uint32_t w, uint32_t par = 0) {
    if (open && gates.size() - steps.back().arg >= kInterpRun - 2) close();
    if (!open) {
      steps.push_back(IStep{I_RUN, (uint32_t)gates.size(), 0, 0});
      open = true;
    }
    gates.push_back(IGate{w, par});
  }
  void close() {
    if (!open) return;
    gates.push_back(IGate{G_END, 0});
    if (gates.size() & 1) gates.push_back(IGate{G_END, 0});
    steps.back().wmask = (uint32_t)gates.size() - steps.back().arg;
    open = false;
  }
};

// One stage's ops.  The signs of a slot are collected until the next square root or H on
// the slot, or the stage's end, as the plan kernels' generator collects them (jit.cpp,
// SignMerge): exact, so both stay bitwise equal.
bool lower_stage(const Plan &P, const DevStage &st, Lowering *L) {
  bool any[kInterpPack + 1] = {};
  uint32_t par[kInterpPack + 1] = {};  // pending signs
  std::vector<IStep> recorded;  // scalar phases and zeroing, applied at the stage's end
  auto scalar = [&](float f, uint32_t q, uint32_t u) { L->step(I_SCALAR, bits_of(f), q, u); };
  auto signed_gate = [&](uint32_t w, int s) {
    L->gate(w, par[s]);
    any[s] = false;
    par[s] = 0;
  };
  for (int i = 0; i < st.op_count; ++i) {
    const DevOp &o = P.ops[st.op_begin + i];
    const int c = o.code;
    if (c < P_DIAG) {
      const int g = (c - P_PAIR) / 6, s = slot_of((c - P_PAIR) % 6);
      if (g == 0) {
        if (any[s]) signed_gate(G_SIGN + s, s);
        L->gate(G_H + s);
        L->gate(G_RS);
      } else {
        signed_gate(((g & 1 ? G_IM : G_RE) + s) | (g >= 3 ? kGateAdj : 0u), s);
      }
    } else if (c < P_CZ) {
      const int d = (c - P_DIAG) / 6, s = slot_of((c - P_DIAG) % 6);
      if (d <= 1) {
        L->gate((G_T + s) | (d ? kGateAdj : 0u) | (o.arg ? kGateUp : 0u));
      } else if (d == 2) {
        if (o.wmask != o.wval || (o.wmask & (o.wmask - 1))) return false;  // (a Z, or a CZ with one fixed qubit)
        any[s] = true;
        par[s] ^= o.wmask ? o.wmask : kParityOne;
      } else {
        L->step(I_MASKMUL, d == 3 ? slot_mask(s) : ~slot_mask(s), o.wmask, o.wval);
      }
    } else if (c < P_PEQ) {
      L->gate(G_CZ + cz_pair((c - P_CZ) / 6, slot_of((c - P_CZ) % 6)));
    } else if (c < P_PHASE) {
      L->step(I_MASKSET, slot_mask((c - P_PEQ) / 6) ^ slot_mask(slot_of((c - P_PEQ) % 6)), o.wmask, o.wval);
    } else if (c == P_PHASE) {
      if (o.arg & 7) recorded.push_back(IStep{I_PHASE, o.arg & 7u, o.wmask, o.wval});
    } else if (c == P_ZERO) {
      recorded.push_back(IStep{I_PHASE, 0, o.wmask, o.wval});
    } else if (c == P_SCALE) {
      scalar(std::ldexp(1.f, -(int)o.arg), 0, 0);
    } else if (c == P_GLOBAL) {
      if (o.arg & 15) scalar(1.f, o.arg & 7u, (o.arg >> 3) & 1u);
    }
  }
  for (int s = 0; s <= kInterpPack; ++s)
    if (any[s]) signed_gate(G_SIGN + s, s);
  for (const IStep &r : recorded) L->step(r.code, r.arg, r.wmask, r.wval);
  if (st.halves || !recorded.empty()) scalar(std::ldexp(1.f, -(int)st.halves), kStageEnd, 0);
  return true;
}

// Whether a stage's lanes cover whole 64-byte runs (or 32-byte halves of one 128-byte row)
// of global memory: tile bit 1 and one of bits 2, 3 are among its five lane bits.
bool lanes_contiguous(const uint8_t *nonr, int group_bits) {
  uint32_t lanes = 0;
  for (int i = 0; i < std::min(group_bits, 5); ++i) lanes |= 1u << nonr[i];
  return (lanes & 2u) && (lanes & 12u);
}

}  // namespace

bool lower_interp(const Plan &P, InterpProgram *out) {
  if (P.layout != 0) return false;
  for (const DevPass &dp : P.passes) {
    const int rk = P.rk, m = dp.m, gb = m - 1 - rk;
    if (!(dp.flags & PF_PACKED) || rk < 1 || rk > kInterpMaxSlots || gb < 1 || gb > 12) return false;
    IHead h;
    std::memset(&h, 0, sizeof(h));
    h.m = dp.m;
    h.flags = dp.flags;
    h.init_amp = dp.init_amp;
    std::memcpy(h.tq, dp.tq, sizeof(dp.tq));
    for (int i = 0; i < dp.nt;) {
      int j = i + 1;
      while (j < dp.nt && dp.ntq[j] == dp.ntq[j - 1] + 1) ++j;
      if (h.runs == 12) return false;
      h.run[h.runs++] = IRun{(uint32_t)((1ull << (j - i)) - 1), (uint8_t)i, dp.ntq[i], 0};
      i = j;
    }
    for (int i = 0; i < 16; ++i)
      for (int b = 0; b < rk; ++b)
        if ((i >> b) & 1) h.it_off[i] |= 1ull << dp.tq[m - rk + b];
    std::vector<IStage> stages;
    Lowering L;
    auto move = [&](uint32_t code, uint32_t arg, uint32_t wval) { L.step(code, arg, 0, wval); };
    const int ns = std::max<int>(dp.stage_count, 1);
    for (int s = 0; s < ns; ++s) {
      IStage is;
      std::memset(&is, 0, sizeof(is));
      uint8_t nonr[12] = {}, rbit[kInterpMaxSlots] = {};
      if (dp.stage_count > 0) {
        const DevStage &st = P.stages[dp.stage_begin + s];
        std::memcpy(nonr, st.nonr, sizeof(nonr));
        std::memcpy(rbit, st.rbit, rk);
      } else {  // a pass without gates (the initial state alone)
        for (int i = 0; i < gb; ++i) nonr[i] = (uint8_t)(1 + i);
        for (int j = 0; j < rk; ++j) rbit[j] = (uint8_t)(m - rk + j);
      }
      auto off = [](int tile_bit) { return 16u * pack_phys(1u << (tile_bit - 1), 0); };
      for (int j = 0; j < rk; ++j) is.reg[j] = off(rbit[j]);
      for (int t = 0; t < 3; ++t)
        for (int v = 0; v < 16; ++v)
          for (int b = 0; b < 4; ++b)
            if (((v >> b) & 1) && 4 * t + b < gb) is.L[16 * t + v] ^= off(nonr[4 * t + b]);
      stages.push_back(is);
      for (int side = 0; side < 2; ++side) {
        if (s != (side ? ns - 1 : 0)) continue;
        uint64_t *g = side ? h.gout : h.gin;
        for (int i = 0; i < gb; ++i) g[i] = 1ull << dp.tq[nonr[i]];
        for (int j = 0; j < rk; ++j) g[12 + j] = 1ull << dp.tq[rbit[j]];
      }
      const bool contiguous = lanes_contiguous(nonr, gb);
      if (s > 0) {
        move(I_LOAD, (uint32_t)s, 0);
      } else if (dp.flags & (PF_INIT_UNIFORM | PF_INIT_ZERO)) {
        move(I_INIT, 0, 0);
      } else if (contiguous) {
        move(I_IN, 0, 0);
      } else {
        move(I_FETCH, 0, 0);
        move(I_LOAD, 0, 1);
      }
      if (dp.stage_count > 0 && !lower_stage(P, P.stages[dp.stage_begin + s], &L)) return false;
      if (s + 1 < ns) {
        move(I_STORE, (uint32_t)s, 0);
      } else if (contiguous) {
        move(I_OUT, 0, 0);
      } else {
        move(I_STORE, (uint32_t)s, 0);
        move(I_SWEEP, 0, 0);
      }
    }
    h.stage_count = (uint32_t)stages.size();
    h.step_count = (uint32_t)L.steps.size();
    h.gate_count = (uint32_t)L.gates.size();
    const size_t o_stage = sizeof(IHead), o_step = o_stage + stages.size() * sizeof(IStage);
    const size_t o_gate = o_step + L.steps.size() * sizeof(IStep);
    const size_t bytes = o_gate + L.gates.size() * sizeof(IGate);
    if (bytes > 0xffffffffull) return false;
    h.bytes = (uint32_t)bytes;
    const size_t at = out->blocks.size();
    out->offset.push_back(at);
    out->bytes.push_back(h.bytes);
    out->blocks.resize(at + h.bytes);
    std::memcpy(&out->blocks[at], &h, sizeof(h));
    std::memcpy(&out->blocks[at + o_stage], stages.data(), stages.size() * sizeof(IStage));
    std::memcpy(&out->blocks[at + o_step], L.steps.data(), L.steps.size() * sizeof(IStep));
    if (!L.gates.empty()) std::memcpy(&out->blocks[at + o_gate], L.gates.data(), L.gates.size() * sizeof(IGate));
  }
  return true;
}

}  // namespace svp
