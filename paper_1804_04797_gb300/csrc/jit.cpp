// Plan-specialised tile-pass kernels: source generation, NVRTC compile, module cache.
#include "jit.h"

#include <cuda.h>
#include <dlfcn.h>
#include <nvrtc.h>
#include <sys/stat.h>
#include <unistd.h>

#include <algorithm>
#include <atomic>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <fstream>
#include <map>
#include <memory>
#include <mutex>
#include <sstream>
#include <thread>
#include <vector>

#include "kernels.h"

namespace svj {

// The device headers, compiled into the library (generated by the build).
extern const int kHeaderCount;
extern const char *const kHeaderNames[];
extern const char *const kHeaderSources[];

namespace {

const char *pair_gate(int g) {
  static const char *names[] = {"GH", "GSX", "GSY", "GSXDG", "GSYDG"};
  return names[g];
}

std::string hex32(uint32_t v) {
  char b[16];
  std::snprintf(b, sizeof(b), "0x%08xu", v);
  return b;
}

// The condition of an op on the thread's condition word W, as a C expression.
std::string cond_expr(const svp::DevOp &o) {
  if (o.wmask == 0) return "true";
  return "((W & " + hex32(o.wmask) + ") == " + hex32(o.wval) + ")";
}

void emit_op(std::ostringstream &os, const svp::DevOp &o) {
  using namespace svp;
  const int c = o.code;
  const std::string C = cond_expr(o);
  os << "      ";
  if (c >= P_PAIR && c < P_PAIR + 30) {
    const int g = (c - P_PAIR) / 6, j = (c - P_PAIR) % 6;
    if (j == kPackSlot) os << "pairs_pack<" << pair_gate(g) << ">(R, I);\n";
    else os << "pairs<" << pair_gate(g) << ", " << j << ">(R, I);\n";
  } else if (c >= P_DIAG && c < P_DIAG + 30) {
    const int d = (c - P_DIAG) / 6, j = (c - P_DIAG) % 6;
    const bool pack = j == kPackSlot;
    if (d <= 1) {  // T or its adjoint, with the plan's rounding constant
      const char *D = d == 0 ? "DT1" : "DTDG1";
      const char *c = o.arg ? "kS2up" : "kS2dn";
      if (pack) os << "diag_pack<" << D << ">(R, I, " << c << ");\n";
      else os << "diag<" << D << ", " << j << ">(R, I, " << c << ");\n";
    } else {
      // Z: sign where the slot is 1; P0: 0 where it is 1; P1: 0 where it is 0
      const int B = d == 4 ? 0 : 1;
      if (d == 2 && !o.wmask) {
        if (pack) os << "negate_pack<1>(R, I);\n";
        else os << "negate<" << j << ", 1>(R, I);\n";
        return;
      }
      const std::string f = d == 2 ? "(" + C + " ? -1.f : 1.f)"
                                   : (o.wmask ? "(" + C + " ? 0.f : 1.f)" : std::string("0.f"));
      if (pack) os << "factor_pack<" << B << ">(R, I, " << f << ");\n";
      else os << "factor<" << j << ", " << B << ">(R, I, " << f << ");\n";
    }
  } else if (c >= P_CZ && c < P_CZ + 36) {
    os << "two<" << (c - P_CZ) / 6 << ", " << (c - P_CZ) % 6 << ", false>(R, I);\n";
  } else if (c >= P_PEQ && c < P_PEQ + 36) {
    os << "two<" << (c - P_PEQ) / 6 << ", " << (c - P_PEQ) % 6 << ", true>(R, I);\n";
  } else if (c == P_PHASE) {
    if (o.wmask) os << "ph += " << C << " ? " << (int)o.arg << " : 0;\n";
    else os << "ph += " << (int)o.arg << ";\n";
  } else if (c == P_ZERO) {
    os << "zero = zero || " << C << ";\n";
  } else if (c == P_SCALE) {
    os << "scale_all(R, I, __int_as_float(" << ((127 - (int)o.arg) << 23) << "));\n";
  } else if (c == P_GLOBAL) {
    if (o.arg & 15) os << "global_factor<" << (o.arg & 7) << ", " << ((o.arg >> 3) & 1) << ">(R, I);\n";
  } else {
    os << "/* no-op */\n";
  }
}

// Signs (Z, and CZ with a qubit outside the register set) on a register slot commute
// with every op except a non-diagonal gate on that slot: the generator collects them per
// slot; their product (an XOR of conditions) rides on the next such gate (its first
// additions become fused operations with y times the sign) or is applied at the end of
// the stage.  Signs are exact, so the result is bitwise the same as applying them one
// by one.
struct SignMerge {
  std::vector<std::string> pend[svp::kPackSlot + 1];
  void add(int j, const std::string &cond) { pend[j].push_back(cond); }
  void flush(std::ostringstream &os, int j) {
    if (pend[j].empty()) return;
    bool all_const = true;
    for (const std::string &c : pend[j]) all_const = all_const && c == "true";
    os << "      ";
    if (all_const) {
      if (pend[j].size() % 2) {
        if (j == svp::kPackSlot) os << "negate_pack<1>(R, I);\n";
        else os << "negate<" << j << ", 1>(R, I);\n";
      } else {
        os << "/* signs cancel */\n";
      }
    } else {
      std::string x;
      for (const std::string &c : pend[j]) x += (x.empty() ? "" : " ^ ") + c;
      const std::string f = "((" + x + ") ? -1.f : 1.f)";
      if (j == svp::kPackSlot) os << "factor_pack<1>(R, I, " << f << ");\n";
      else os << "factor<" << j << ", 1>(R, I, " << f << ");\n";
    }
    pend[j].clear();
  }
  void flush_all(std::ostringstream &os) {
    for (int j = 0; j <= svp::kPackSlot; ++j) flush(os, j);
  }
  // The pending signs of slot j as the sign argument of the next gate on it: "" when
  // they cancel, else a C expression (+1 or -1); clears them.
  std::string take(int j) {
    std::string r;
    if (pend[j].empty()) return r;
    bool all_const = true;
    for (const std::string &c : pend[j]) all_const = all_const && c == "true";
    if (all_const) {
      r = pend[j].size() % 2 ? "-1.f" : "";
    } else {
      std::string x;
      for (const std::string &c : pend[j]) x += (x.empty() ? "" : " ^ ") + c;
      r = "((" + x + ") ? -1.f : 1.f)";
    }
    pend[j].clear();
    return r;
  }
};

// The ops of one stage.  The factors 1/2 the stage leaves pending at its end
// (DevStage::halves) are added to *halves for the caller to apply later.  fuse_phase: a T
// (or its adjoint) on a register slot waits, like the signs, for the next gate on that
// slot and is applied with it (pairs_diag), else at the end of the stage; the result
// differs from applying it in place by rounding only.  The planner places each T of these
// plans in the stage of the next gate on its qubit (plan.cpp), so it nearly always rides
// on one: 34-qubit circuit 0.380 s -> 0.374 s with the T ops where they fell (29 of 69
// fused), 0.362 s with them placed (39 fused; the others are phases of the tile or have no
// later gate).  Off for the kernels that must match the interpreter bit for bit.
void emit_stage_ops(std::ostringstream &os, const svp::Plan &P, const svp::DevStage &st, int *halves,
                    bool fuse_phase = false) {
  using namespace svp;
  SignMerge signs;
  const DevOp *tpend[kPackSlot + 1] = {};  // the waiting T op of each slot
  for (int o = 0; o < st.op_count; ++o) {
    const DevOp &op = P.ops[st.op_begin + o];
    const int c = op.code;
    if (c >= P_PAIR && c < P_PAIR + 30) {
      // the slot's pending signs ride on the gate's first additions
      const int g = (c - P_PAIR) / 6, j = (c - P_PAIR) % 6;
      const std::string sg = signs.take(j);
      if (tpend[j]) {
        const int d = (tpend[j]->code - P_DIAG) / 6;
        const std::string k = tpend[j]->arg ? "kS2up" : "kS2dn";
        const std::string sc = sg.empty() ? k : "(" + sg + ") * " + k;
        const char *D = d == 0 ? "DT1" : "DTDG1";
        if (j == kPackSlot) os << "      pairs_pack_diag<" << pair_gate(g) << ", " << D << ">(R, I, " << sc << ");\n";
        else os << "      pairs_diag<" << pair_gate(g) << ", " << D << ", " << j << ">(R, I, " << sc << ");\n";
        tpend[j] = nullptr;
        continue;
      }
      if (!sg.empty()) {
        if (j == kPackSlot) os << "      pairs_pack_signed<" << pair_gate(g) << ">(R, I, " << sg << ");\n";
        else os << "      pairs_signed<" << pair_gate(g) << ", " << j << ">(R, I, " << sg << ");\n";
        continue;
      }
    } else if (c >= P_DIAG + 12 && c < P_DIAG + 18) {  // Z on a slot (conditional or not)
      signs.add((c - P_DIAG) % 6, cond_expr(op));
      continue;
    } else if (fuse_phase && c >= P_DIAG && c < P_DIAG + 12) {  // T or its adjoint on a slot
      const int j = (c - P_DIAG) % 6;
      if (tpend[j]) emit_op(os, *tpend[j]);  // a second one: the first in place
      tpend[j] = &op;
      continue;
    } else if (c >= P_U && c < P_U + 6 && tpend[c - P_U]) {  // a general gate on the slot
      emit_op(os, *tpend[c - P_U]);
      tpend[c - P_U] = nullptr;
    }
    emit_op(os, op);
  }
  for (const DevOp *t : tpend)
    if (t) emit_op(os, *t);
  signs.flush_all(os);
  *halves += st.halves;
}

// The end of a stage: the recorded zeroing, scalar phase and the exact factors 1/2 that
// are due.  A stage's pending factors 1/2 (pairs of the square roots' 2^{-1/2}) wait for a
// later stage end (an exact power-of-two scale); at most kCarry are carried into a stage,
// which itself scales after every kMaxDeferred of them, so values stay below
// 2^(kCarry + kMaxDeferred + 1).
void emit_stage_end(std::ostringstream &os, int *pending, bool last_of_pass) {
  constexpr int kCarry = 32;
  int now = 0;
  if (*pending > kCarry || last_of_pass) {
    now = *pending;
    *pending = 0;
  }
  while (now > svp::kMaxDeferred) {
    os << "      scale_all(R, I, __int_as_float(" << ((127 - svp::kMaxDeferred) << 23) << "));\n";
    now -= svp::kMaxDeferred;
  }
  os << "      end_stage(R, I, " << now << ", ph, zero);\n";
}

// The qubits on which pass `pass` may find amplitudes other than those of its starting basis
// state: the tiles' qubits of the passes before it (every qubit for other plans).
uint64_t support(const svp::Plan &P, int pass) {
  if (!P.basis) return ~0ull;
  uint64_t u = 0;
  for (int k = 0; k < pass; ++k)
    for (int i = 0; i < P.passes[(size_t)k].m; ++i) u |= 1ull << P.passes[(size_t)k].tq[i];
  return u;
}

// Where qubit q's bit lies in the state a plan's kernels address: a plan from a basis state
// keeps the amplitudes its passes write and no others -- the support that its last pass, which
// stores nothing, finds -- in index order (-1: not a bit of it).
int place(const svp::Plan &P, int q) {
  if (!P.basis) return q;
  const uint64_t U = support(P, (int)P.passes.size() - 1);
  return (U >> q) & 1ull ? __builtin_popcountll(U & ((1ull << q) - 1)) : -1;
}
uint64_t placed(const svp::Plan &P, uint64_t index) {
  if (!P.basis) return index;
  uint64_t v = 0;
  for (; index; index &= index - 1) {
    const int at = place(P, __builtin_ctzll(index));
    if (at >= 0) v |= 1ull << at;
  }
  return v;
}

// The tile index bits of the last pass at which the qubits of Plan::all_of lie.
uint64_t listed_bits(const svp::Plan &P) {
  const svp::DevPass &dp = P.passes.back();
  uint64_t v = 0;
  for (int i = 0; i < dp.nt; ++i) v |= ((P.all_of >> dp.ntq[i]) & 1ull) << i;
  return v;
}

// C expression of a stage's group addressing for thread index `var`: the XOR over its
// group-index bits of the stage's per-bit offsets (L: shared-memory byte offset, 32-bit;
// G: global index offset, 64-bit; `whole`: in the whole state, where P's is kept compactly), as
// compile-time constants -- no table reads.
std::string group_expr(const svp::Plan &P, uint32_t si, const char *var, bool global, bool whole = false) {
  const svp::DevStage &st = P.stages[si];
  (void)st;
  const svp::DevGroupEntry *ge = &P.gtab[(size_t)svp::kGroupEntries * si];
  std::string e;
  for (int i = 0; i < 12; ++i) {
    // bit i of the group index is entry (1 << (i % 4)) of table i / 4
    const svp::DevGroupEntry &x = ge[16 * (i / 4) + (1 << (i % 4))];
    const uint64_t v = !global ? (uint64_t)x.L : whole ? x.G : placed(P, x.G);
    if (!v) continue;
    char b[96];
    if (global) std::snprintf(b, sizeof(b), "((%s >> %d) & 1 ? 0x%llxull : 0ull)", var, i, (unsigned long long)v);
    else std::snprintf(b, sizeof(b), "((%s >> %d) & 1 ? 0x%xu : 0u)", var, i, (unsigned)v);
    e += (e.empty() ? "" : " ^ ") + std::string(b);
  }
  return e.empty() ? (global ? "0ull" : "0u") : e;
}

// C expression of the global index of tile `tile_id`'s element 0: the tile index bits
// spread over the non-tile qubits, one shift-and-mask per run of consecutive qubits.  (whole: in
// the whole state, where P's is kept compactly)
std::string tile_base_expr(const svp::Plan &P, const svp::DevPass &dp, bool whole = false) {
  std::string e;
  auto at = [&](int i) { return whole ? (int)dp.ntq[i] : place(P, dp.ntq[i]); };
  for (int i = 0; i < dp.nt;) {
    int j = i + 1;
    if (at(i) < 0) { i = j; continue; }
    while (j < dp.nt && at(j) == at(j - 1) + 1) ++j;
    char b[160];
    std::snprintf(b, sizeof(b), "((tile_id >> %d) & 0x%llxull) << %d", i, (unsigned long long)((1ull << (j - i)) - 1),
                  at(i));
    e += (e.empty() ? "" : " | ") + std::string("(") + b + ")";
    i = j;
  }
  return e.empty() ? "0ull" : e;
}

}  // namespace

int register_slots() {
  // SV_REG_SLOTS (3..5) overrides the register slots of the plan-specialised kernels
  // (tuning: 5 = 64 amplitudes a thread, stages of six qubits)
  static int slots = [] {
    const char *e = std::getenv("SV_REG_SLOTS");
    const int v = e ? std::atoi(e) : 0;
    return (v >= 3 && v <= 5) ? v : kRegisterSlots;
  }();
  return slots;
}

// Log2 of the runs of neighbouring tiles a CTA of a pipelined kernel takes per turn of the
// grid (tile_of in tile_pipe.cuh).  SV_TILE_RUN (0..3) overrides it (tuning).
int tile_run_log() {
  static int v = [] {
    const char *e = std::getenv("SV_TILE_RUN");
    const int x = e ? std::atoi(e) : -1;
    return (x >= 0 && x <= 3) ? x : kTileRunLog;
  }();
  return v;
}

bool pipe_shape(int m, int *groups, int *slots) {
  if (m < 10 || m > 13) return false;  // a group is at least one warp (named barriers)
  // groups x slots per tile size; SV_PIPE_SHAPE="G,S" overrides the 12- and 13-qubit
  // shapes (tuning: 1..8 groups, slots a multiple of the groups and within shared memory).
  // Group g owns slots g, g + G, ...: every slot is filled and emptied in one order, so
  // a wait on a slot's mbarrier is never more than one phase ahead of it (the parity
  // wait could not tell phase k from phase k - 2).
  static int env_g = -1, env_s = -1;
  static std::once_flag once;
  std::call_once(once, [] {
    const char *e = std::getenv("SV_PIPE_SHAPE");
    int g = 0, s = 0;
    if (e && std::sscanf(e, "%d,%d", &g, &s) == 2 && g >= 1 && g <= 8 && s >= g && s % g == 0) {
      env_g = g;
      env_s = s;
    }
  });
  int g = m <= 11 ? 4 : m == 12 ? kPipeGroups12 : 1;
  int s = m <= 11 ? 8 : m == 12 ? kPipeSlots12 : 3;
  if (m >= 12 && env_g > 0 && (size_t)env_s * (sizeof(float2) << m) + 2048 <= 227 * 1024 &&
      env_g * (1 << (m - 5)) + 32 <= 1024) {
    g = env_g;
    s = env_s;
  }
  *groups = g;
  *slots = s;
  return true;
}

int pass_matrix_stages(const svp::Plan &P, int pass) {
  if (!P.mma) return 0;
  const svp::DevPass &dp = P.passes[(size_t)pass];
  int k = 0;
  for (uint32_t s = 0; s < dp.stage_count; ++s) k += P.stage_gates[dp.stage_begin + s].empty() ? 0 : 1;
  return k;
}

size_t pass_mma_smem(const svp::Plan &P, int pass) {
  // two B buffers, each one stage's hi and lo parts (64 x 64, fp16 or fp32)
  return pass_matrix_stages(P, pass) > 0 ? (size_t)2 * 2 * 64 * 64 * (P.mma == 1 ? 2 : 4) : 0;
}

// SV_MMA_SHAPE "G,S" overrides the compute groups and slots of a tensor-core pass (tuning: within
// TMEM, shared memory and threads, S a multiple of G).
namespace {
struct MmaShape {
  int g = 0, s = 0;
};
MmaShape mma_shape_env(int mma) {
  static MmaShape env[3];
  static std::once_flag once;
  std::call_once(once, [] {
    const char *e = std::getenv("SV_MMA_SHAPE");
    int g = 0, s = 0;
    if (e && std::sscanf(e, "%d,%d", &g, &s) == 2 && g >= 1 && s >= g && s % g == 0)
      for (int k = 1; k <= 2; ++k) {
        const int cols = k == 1 ? 128 : 256;
        const size_t smem = (size_t)s * 32768 + 2 * 2 * 64 * 64 * (k == 1 ? 2 : 4) + 1024;
        if (g * cols <= 512 && smem <= 216 * 1024 && g * 128 + 96 <= 1024) env[k] = MmaShape{g, s};
      }
  });
  return env[mma];
}
}  // namespace

bool pass_pipe_shape(const svp::Plan &P, int pass, int *groups, int *slots) {
  const int m = P.passes[(size_t)pass].m;
  if (pass_matrix_stages(P, pass) > 0) {
    const MmaShape e = mma_shape_env(P.mma);
    if (m == 12 && e.g) {
      *groups = e.g;
      *slots = e.s;
      return true;
    }
    // tensor-core passes (12-qubit tiles): groups of four warps, each with a tile in flight.
    // TF32x3 two (2 x 256 TMEM columns of A hi, A lo and D); F16x3 (128 columns) four where the
    // CTAs have several tiles each -- a group's instructions wait for one another, so more warps
    // fill the issue slots although 96 registers spill a little -- and two below that (us at 2 / 4
    // groups, one GB300: 12 qubits 13.9 / 15.7, 16 32.7 / 33.2, 19 36.3 / 37.3, 20 43.0 / 45.0,
    // 21 63.8 / 59.8, 22 102 / 88; two tiles in flight for each of two groups, as it was: 14.3,
    // 32.0, 35.9, 47.8, 62.0, 93.4; 25 qubits 728 -> 696, 28 3.38 -> 3.25 ms, 32 71.4 -> 67.3).
    // Shared memory: four 32 KB slots and two B buffers (2 x 16 KB or 2 x 32 KB).
    if (m != 12) return false;
    *groups = P.mma == 1 && P.n >= 21 ? 4 : 2;
    *slots = 4;
    return true;
  }
  if (!pipe_shape(m, groups, slots)) return false;
  // the plan's groups for the pass, with the slots cut to a multiple of them (12-qubit
  // tiles: 3 or 2 groups on six slots, 4 on four)
  const int g = (size_t)pass < P.pipe_groups.size() ? P.pipe_groups[(size_t)pass] : 0;
  if (g > 0 && *slots >= g && g * (1 << (m - 5)) + 64 <= 1024) {
    *groups = g;
    *slots -= *slots % g;
  }
  return true;
}

// Whether the last stage of pass `pass` holds whole 128-byte rows per quarter warp (its
// three lane bits are tile bits 1..3): then its registers go straight to HBM.
bool pipe_direct_store(const svp::Plan &P, int pass) {
  const svp::DevPass &dp = P.passes[(size_t)pass];
  if (dp.stage_count == 0) return false;
  // the plain kernels' write-only first pass is bound by its arithmetic: its groups hand
  // the stores to the storer warp's TMA copies instead of waiting on their own (34 qubits:
  // 57 -> 50 ms; the read-write passes measured the same either way; the tensor-core
  // passes measured slower: F16x3 pass 0 166 -> 174 ms)
  if ((dp.flags & (svp::PF_INIT_UNIFORM | svp::PF_INIT_ZERO)) && pass_matrix_stages(P, pass) == 0) return false;
  const svp::DevStage &ls = P.stages[dp.stage_begin + dp.stage_count - 1];
  int mask = 0;
  for (int i = 0; i < 3; ++i) mask |= 1 << ls.nonr[i];
  return mask == ((1 << 1) | (1 << 2) | (1 << 3));
}

int pipe_threads(const svp::Plan &P, int kpr, int pass, bool inner) {
  int G = 0, S = 0;
  const svp::DevPass &dp = P.passes[(size_t)pass];
  if (!pass_pipe_shape(P, pass, &G, &S)) return 0;
  const bool last = (size_t)pass + 1 == P.passes.size();
  const bool direct = (inner && last) || pipe_direct_store(P, pass);
  return G * (1 << (dp.m - 1 - kpr)) + 32 + (direct ? 0 : 32) + (pass_matrix_stages(P, pass) > 0 ? 32 : 0);
}

// Stages of a pass with matrix stages whose tile offsets lie in a shared-memory table (256 bytes
// each) instead of being put together from the thread's index at every use (about 20 instructions,
// twice a stage and tile; with the mixed-precision split, 28 qubits F16x3 7.76 -> 7.67 ms).
constexpr int kOffsetStages = 32;

std::string pipe_pass_source(const svp::Plan &P, int kpr, int pass, bool inner) {
  const svp::DevPass &dp = P.passes[(size_t)pass];
  const int m = dp.m;
  int G = 0, S = 0;
  if (!pass_pipe_shape(P, pass, &G, &S) || S % G != 0) return std::string("#error \"no pipelined shape for this tile\"\n");
  const int TG = 1 << (m - 1 - kpr);             // threads of one compute group
  const int nbox = 1 << (m - 7);                  // 1 KB boxes (8 rows of 128 B) per tile
  const bool init = (dp.flags & (svp::PF_INIT_UNIFORM | svp::PF_INIT_ZERO)) != 0;
  const bool last = (size_t)pass + 1 == P.passes.size();
  inner = inner && last;
  // a plan from a basis state: the tile index bits that take both values (the others are
  // x's), and whether tile qubits outside the support leave most of the tile zero -- the
  // first stage then reads the rest itself, straight into its registers
  const uint64_t U = support(P, pass);
  uint64_t vary = 0;
  bool masked = false;
  for (int i = 0; i < dp.nt; ++i) vary |= ((U >> dp.ntq[i]) & 1ull) << i;
  for (int i = 0; i < m; ++i) masked = masked || !((U >> dp.tq[i]) & 1ull);
  const bool all_tiles = vary == (dp.nt >= 64 ? ~0ull : (1ull << dp.nt) - 1);
  const bool fork = P.fork > 0 && pass == 0;  // reads the prefix, scaled (Plan::fork)
  // the listed tiles alone (Plan::listed)
  const bool listed = last && P.listed;
  // C statements: this CTA's tile of turn i (leaves the loop after the last one)
  const std::string this_tile = [&]() {
    const std::string id = all_tiles && !fork && !listed ? "tile_id" : "tile_j";
    std::string t = "const unsigned long long " + id + " = tile_of<RUN>(i, num_tiles);\n      if (" + id +
                    " >= num_tiles) break;\n";
    if (id == "tile_id") return t;
    if (fork) return t + "      const unsigned long long tile_id = first_tile + tile_j;\n";
    uint64_t bits = vary;  // the tile index bits that tile_j runs through
    if (listed) bits = listed_bits(P);
    t += listed ? "      const unsigned long long tile_id = __ldg(tile_list + (tile_j >> " +
                      std::to_string(__builtin_popcountll(bits)) + "))"
                : std::string("      const unsigned long long tile_id = ba.fixed");
    for (int i = 0, from = 0; i < dp.nt;) {
      if (!((bits >> i) & 1ull)) { ++i; continue; }
      int k = i;
      while (k < dp.nt && ((bits >> k) & 1ull)) ++k;
      t += " | (((tile_j >> " + std::to_string(from) + ") & " + std::to_string((1ull << (k - i)) - 1) + "ull) << " +
           std::to_string(i) + ")";
      from += k - i;
      i = k;
    }
    return t + ";\n      (void)tile_id;\n";
  }();
  // the last stage's output: straight from registers (whole rows per quarter warp), or
  // back into the slot in memory order, written out by a storer warp with TMA stores
  const bool direct = inner || pipe_direct_store(P, pass);
  const int NT = pipe_threads(P, kpr, pass, inner);
  // tensor-core matrix stages (fused packed plans): an MMA warp after the other roles
  const int nms = pass_matrix_stages(P, pass);
  const bool mma = nms > 0;
  if (mma && (kpr != 4 || TG != 128 || inner || S % G != 0))
    return std::string("#error \"matrix stages need 12-qubit tiles and four register slots\"\n");
  const bool f16 = P.mma == 1;
  const bool restore = mma && (dp.flags & svp::PF_UNITARY) && !(dp.flags & svp::PF_RAW);
  const int MT0 = G * TG + 32 + (direct ? 0 : 32);  // first thread of the MMA warp
  auto row_of = [&](int q) { return place(P, q) < 4 ? 0u : 1u << (place(P, q) - 4); };
  std::string boxrow;  // C statements: row += the row offset of box j
  for (int b = 0; b + 7 < m; ++b)
    boxrow += "        if ((j >> " + std::to_string(b) + ") & 1) row += " + std::to_string(row_of(dp.tq[7 + b])) + ";\n";
  std::ostringstream os;
  // the fork's scaling of a loaded group, as fork_kernel does it, operation by operation
  auto emit_fork_scale = [&]() {
    const svk::ForkScale f = svk::fork_scale(P.fork);
    char hi[32], lo[32];
    std::snprintf(hi, sizeof(hi), "%.9ef", f.hi);
    std::snprintf(lo, sizeof(lo), "%.9ef", f.lo);
    auto scaled = [&](const std::string &v) {
      return f.lo == 0.f ? v + " * " + hi : "fmaf(" + v + ", " + hi + ", " + v + " * " + lo + ")";
    };
    os << "#pragma unroll\n      for (int p = 0; p < kP; ++p) {\n"
       << "        R[p] = f2(" << scaled("R[p].x") << ", " << scaled("R[p].y") << ");\n"
       << "        I[p] = f2(" << scaled("I[p].x") << ", " << scaled("I[p].y") << ");\n      }\n";
  };
  os << "// pipelined tile-pass kernel of one pass of a plan\n#define SV_PACK_R " << kpr
     << "\n#include \"tile_pack.cuh\"\n#include \"tile_pipe.cuh\"\n"
     << (mma ? "#include \"tile_mma.cuh\"\n" : "")
     << "using namespace svk::tpk;\nusing namespace svk::tpipe;\n" << (mma ? "using namespace svk::tmma;\n" : "");
  if (mma) {
    // byte offset in the plan's matrices of each matrix stage's B (hi part, then lo)
    os << "\n__device__ __forceinline__ unsigned long long b_src(int s) {\n  switch (s) {\n";
    int k = 0;
    for (uint32_t st = 0; st < dp.stage_count; ++st) {
      const uint32_t si = dp.stage_begin + st;
      if (P.stage_gates[si].empty()) continue;
      os << "    case " << k++ << ": return " << (unsigned long long)P.stages[si].mat_begin * 4ull << "ull;\n";
    }
    os << "    default: return 0ull;\n  }\n}\n";
  }
  os << "\nextern \"C\" __global__ void __launch_bounds__(" << NT << ", 1)\nsv_pass"
     << "(float2 *__restrict__ psi, svk::DevPlanView plan, unsigned long long num_tiles, double *sums,\n"
     << "        const float2 *__restrict__ other, const __grid_constant__ TmaDesc tmap"
     << (P.basis ? ", const svk::BasisArgs ba" : fork ? ", const unsigned long long first_tile"
         : listed ? ", const unsigned long long *__restrict__ tile_list" : "") << ") {\n"
     << "  constexpr int G = " << G << ", S = " << S << ", TG = " << TG << ";\n"
     << "  constexpr int RUN = " << (mma ? 0 : tile_run_log()) << ";  // runs of 2^RUN neighbouring tiles per turn\n"
     << "  constexpr unsigned TILE_BYTES = " << (8u << m) << "u;\n"
     << "  extern __shared__ __align__(1024) unsigned char smem_raw[];\n"
     << "  // full: a tile has landed in the slot; empty: the slot may be reloaded" << (direct ? "" : ";\n"
        "  // done: the slot holds a finished tile (in memory order) to write out") << "\n"
     << "  __shared__ __align__(8) unsigned long long full_bar[S], empty_bar[S]" << (direct ? "" : ", done_bar[S]")
     << ";\n"
     << "  __shared__ svp::DevPass P;\n"
     << "  // slots on a 1 KB boundary (the copies' 128-byte swizzle repeats every 1 KB)\n"
     << "  unsigned char *smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);\n"
     << "  const int tid = threadIdx.x;\n";
  if (mma) {
    os << "  constexpr int NMS = " << nms << ";                // matrix stages of the pass\n"
       << "  constexpr unsigned BSTAGE = " << 2 * 64 * 64 * (f16 ? 2 : 4) << "u;  // one stage's B (hi + lo)\n"
       << "  constexpr uint32_t ACOLS = " << (f16 ? 32 : 64) << "u, CG = " << (f16 ? 128 : 256)
       << "u;  // TMEM columns: one A part; one group (A hi, A lo, D)\n"
       << "  constexpr int MT0 = " << MT0 << ";  // the MMA warp\n"
       << "  unsigned char *bring = smem + S * TILE_BYTES;  // two B buffers\n"
       << "  // a_full[g]: group g's A is in TMEM; d_full[g]: its products are done; b_full /\n"
       << "  // b_free: a B buffer has landed / its products have read it\n"
       << "  __shared__ __align__(8) unsigned long long a_full[G], d_full[G], b_full[2], b_free[2], drain_bar;\n"
       << "  __shared__ uint32_t tmem_base;\n";
    if (restore || f16)
      os << "  __shared__ float2 nrm[2][G][2][4];  // per tile parity and group: warp sums of the norm in / out\n";
  }
  os << "  if (tid == 0) {\n"
     << "    P = plan.passes[" << pass << "];\n"
     << "    for (int s = 0; s < S; ++s) {\n"
     << "      mbar_init(&full_bar[s], 1);\n";
  if (direct) os << "      mbar_init(&empty_bar[s], TG);\n";
  else os << "      mbar_init(&empty_bar[s], 1);\n      mbar_init(&done_bar[s], TG);\n";
  os << "    }\n";
  if (mma)
    os << "    for (int g = 0; g < G; ++g) { mbar_init(&a_full[g], TG); mbar_init(&d_full[g], 1); }\n"
       << "    for (int b = 0; b < 2; ++b) { mbar_init(&b_full[b], 1); mbar_init(&b_free[b], 1); }\n"
       << "    mbar_init(&drain_bar, 1);\n";
  os << "    mbar_init_fence();\n"
     << "  }\n";
  // matrix stages: each thread's byte offset in the tile (below 32 KB), by stage
  const bool table = mma && dp.stage_count <= kOffsetStages;
  if (table) {
    os << "  __shared__ unsigned short a0_tab[" << dp.stage_count << "][TG];\n  if (tid < TG) {\n    const int t = tid;\n";
    for (uint32_t st = 0; st < dp.stage_count; ++st)
      os << "    a0_tab[" << st << "][t] = (unsigned short)(" << group_expr(P, dp.stage_begin + st, "t", false) << ");\n";
    os << "  }\n";
  }
  if (mma)
    os << "  if (tid >= MT0) {  // the MMA warp holds the CTA's tensor memory (one CTA per SM)\n"
       << "    asm volatile(\"tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\" ::\"r\"(smem_u32(&tmem_base)));\n"
       << "    asm volatile(\"tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\");\n"
       << "  }\n"
       << "  fence_before();\n  __syncthreads();\n  fence_after();\n"
       << "  const uint32_t tmem = tmem_base;\n";
  else
    os << "  __syncthreads();\n";
  os << "  double a2 = 0.0, a4 = 0.0;\n"
     << "  (void)sums; (void)other; (void)tmap;\n"
     << "  const int lane = tid & 31;\n"
     << "  if (tid >= G * TG && tid < G * TG + 32) {\n"
     << "    // producer warp: tile i of this CTA into slot i mod S once the slot is empty\n"
     << "    unsigned long long i = 0;\n"
     << "    for (;; ++i) {\n"
     << "      " << this_tile
     << "      const int s = (int)(i % S);\n"
     << "      bool ok = i < S || mbar_wait(&empty_bar[s], (uint32_t)((i / S - 1) & 1), kWaitNs);\n"
     << "      ok = __all_sync(0xffffffffu, ok);\n"
     << "      if (!ok) { if (lane == 0) atomicExch(plan.err, 3); break; }\n";
  if (init || masked) {
    os << "      if (lane == 0) mbar_arrive(&full_bar[s]);  // "
       << (init ? "generated tile: nothing to read" : "read by the first stage") << "\n";
  } else {
    os << "      if (lane == 0) mbar_arrive_tx(&full_bar[s], TILE_BYTES);\n"
       << "      __syncwarp();\n"
       << "      const int row0 = (int)(((" << tile_base_expr(P, dp) << ")"
       << (fork ? " & " + std::to_string((1ull << (P.n - P.fork)) - 1) + "ull" : std::string()) << ") >> 4);\n"
       << "      unsigned char *dst = smem + s * TILE_BYTES;\n"
       << "      for (int j = lane; j < " << nbox << "; j += 32) {\n"
       << "        int row = row0;\n"
       << boxrow
       << "        tma_load_5d(dst + j * 1024, &tmap, 0, 0, 0, 0, row, &full_bar[s]);\n"
       << "      }\n";
  }
  os << "    }\n";
  if (!init && !masked)
    os << "    // every issued copy has landed before the CTA exits (bounded)\n"
       << "    for (unsigned long long k = i > (unsigned long long)S ? i - S : 0; k < i; ++k)\n"
       << "      mbar_wait(&full_bar[k % S], (uint32_t)((k / S) & 1), kWaitNs);\n";
  if (mma) {
    os << "  } else if (tid >= MT0) {\n"
       << "    // MMA warp: for each round of G tiles (group g's tile j G + g), each matrix stage s\n"
       << "    // and each group g, wait for the group's A and issue its products with stage s's B;\n"
       << "    // B is streamed from the plan into two buffers one stage ahead.\n"
       << "    if (elect_lane()) {\n"
       << "      const unsigned long long mine = tiles_of_cta<RUN>(num_tiles);\n"
       << "      const unsigned long long rounds = (mine + G - 1) / G, steps = rounds * NMS;\n"
       << "      const unsigned char *bsrc = reinterpret_cast<const unsigned char *>(plan.mats);\n"
       << "      uint32_t apar = 0;\n"
       << "      bool ok = true;\n"
       << "      unsigned long long q = 0, loaded = 0, landed = 0;\n"
       << "      if (steps > 0) {\n"
       << "        mbar_arrive_tx(&b_full[0], BSTAGE);\n"
       << "        bulk_g2s(bring, bsrc + b_src(0), BSTAGE, &b_full[0]);\n"
       << "        loaded = 1;\n"
       << "      }\n"
       << "      for (unsigned long long j = 0; ok && j < rounds; ++j) {\n"
       << "        for (int s = 0; ok && s < NMS; ++s, ++q) {\n"
       << "          const int buf = (int)(q & 1);\n"
       << "          if (!mbar_wait(&b_full[buf], (uint32_t)((q >> 1) & 1), kWaitNs)) { ok = false; break; }\n"
       << "          ++landed;\n"
       << "          const uint32_t bh = smem_u32(bring + buf * BSTAGE), bl = bh + BSTAGE / 2;\n"
       << "          for (int g = 0; g < G; ++g) {\n"
       << "            if (j * G + g >= mine) continue;\n"
       << "            if (!mbar_wait(&a_full[g], (apar >> g) & 1u, kWaitNs)) { ok = false; break; }\n"
       << "            apar ^= 1u << g;\n"
       << "            fence_after();\n"
       << "            issue_products<" << (f16 ? "true" : "false")
       << ">(tmem + g * CG + 2 * ACOLS, tmem + g * CG, tmem + g * CG + ACOLS, bh, bl);\n"
       << "            mma_commit(&d_full[g]);\n"
       << "            // the next step's B into the other buffer, as soon as the products of the\n"
       << "            // step before this one have left it: behind this step's first products\n"
       << "            // (at the step's end its latency was exposed: 28 qubits F16x3 8.11 -> 7.93 ms,\n"
       << "            // 25 qubits TF32x3 1.14 -> 1.10 ms)\n"
       << "            if (g == 0 && q + 1 < steps) {\n"
       << "              if (q >= 1 && !mbar_wait(&b_free[buf ^ 1], (uint32_t)(((q - 1) >> 1) & 1), kWaitNs)) { ok = false; break; }\n"
       << "              mbar_arrive_tx(&b_full[buf ^ 1], BSTAGE);\n"
       << "              bulk_g2s(bring + (buf ^ 1) * BSTAGE, bsrc + b_src((s + 1) % NMS), BSTAGE, &b_full[buf ^ 1]);\n"
       << "              ++loaded;\n"
       << "            }\n"
       << "          }\n"
       << "          if (!ok) break;\n"
       << "          mma_commit(&b_free[buf]);\n"
       << "        }\n"
       << "      }\n"
       << "      // every product issued has completed and every B copy issued has landed (bounded)\n"
       << "      mma_commit(&drain_bar);\n"
       << "      mbar_wait(&drain_bar, 0, kWaitNs);\n"
       << "      for (unsigned long long k = landed; k < loaded; ++k) mbar_wait(&b_full[k & 1], (uint32_t)((k >> 1) & 1), kWaitNs);\n"
       << "      if (!ok) atomicExch(plan.err, 4);\n"
       << "    }\n"
       << "    __syncwarp();\n";
  }
  if (!direct) {
    os << "  } else if (tid >= G * TG + 32) {\n"
       << "    // storer warp: tile i out of its slot once its group has written it back, then\n"
       << "    // the slot goes to the producer\n"
       << "    for (unsigned long long i = 0;; ++i) {\n"
       << "      " << this_tile
       << "      const int s = (int)(i % S);\n"
       << "      bool ok = mbar_wait(&done_bar[s], (uint32_t)((i / S) & 1), kWaitNs);\n"
       << "      ok = __all_sync(0xffffffffu, ok);\n"
       << "      if (!ok) { if (lane == 0) atomicExch(plan.err, 3); break; }\n"
       << "      const int row0 = (int)((" << tile_base_expr(P, dp) << ") >> 4);\n"
       << "      const unsigned char *src = smem + s * TILE_BYTES;\n"
       << "      for (int j = lane; j < " << nbox << "; j += 32) {\n"
       << "        int row = row0;\n"
       << boxrow
       << "        tma_store_5d(&tmap, 0, 0, 0, 0, row, src + j * 1024);\n"
       << "      }\n"
       << "      bulk_commit();\n"
       << "      bulk_wait_read_all();  // the slot has been read out\n"
       << "      __syncwarp();\n"
       << "      if (lane == 0) mbar_arrive(&empty_bar[s]);\n"
       << "    }\n"
       << "    bulk_wait_all();  // the stores have completed before the CTA exits\n";
  }
  if (mma) {
    // ---- compute groups with tensor-core matrix stages
    os << "  } else {\n"
       << "    // group g takes tiles g, g + G, ...: tile i in slot i mod S (S a multiple of G).  One\n"
       << "    // group's products run while the others work.\n"
       << "    const int g = tid / TG, t = tid % TG;\n"
       << "    const int bar_id = 1 + g;\n"
       << "    const uint32_t tl = tmem + ((uint32_t)(32 * ((tid >> 5) & 3)) << 16);  // this thread's TMEM lane\n"
       << "    Regs R, I;\n"
       << "    const uint32_t tg = tl + (uint32_t)g * CG;\n"
       << "    for (unsigned long long i = (unsigned long long)g, k = 0;; i += G, ++k) {\n"
       << "      " << this_tile
       << "      const int slot = (int)(i % S);\n"
       << "      float4 *tile = reinterpret_cast<float4 *>(smem + slot * TILE_BYTES);\n"
       << "      const uint32_t W = ((uint32_t)tile_id << " << (m - 1 - kpr) << ") | (uint32_t)t;\n"
       << "      float sc = 1.f;   // F16: the tile's scale (power of two) from its first product\n"
       << "      bool okm = true;  // every product wait of the tile succeeded\n"
       << "      (void)W; (void)sc;\n";
    const int ns = dp.stage_count;
    // matrix-stage index of each stage (-1: no products), and the first one
    std::vector<int> msi(ns, -1);
    int first_ms = -1;
    for (int s = 0, q = 0; s < ns; ++s)
      if (!P.stage_gates[dp.stage_begin + (uint32_t)s].empty()) {
        msi[s] = q++;
        if (first_ms < 0) first_ms = s;
      }
    int pending = 0;  // factors 1/2 pending (lowered square roots only; none in these plans)
    auto stage_head = [&](uint32_t si) {
      os << "        const uint32_t rx[" << kpr << "] = {";
      for (int j = 0; j < kpr; ++j)
        os << (j ? ", " : "") << hex32(P.gtab[(size_t)svp::kGroupEntries * si + svp::kRegEntry + j].L);
      os << "};\n";
      if (table) {
        os << "        const uint32_t a0 = a0_tab[" << si - dp.stage_begin << "][t];\n";
        return;
      }
      // (recomputed at every use: hoisted out of the tile loop, every stage's address
      // would stay live and spill)
      os << "        uint32_t a0 = " << group_expr(P, si, "t", false) << ";\n"
         << "        asm volatile(\"\" : \"+r\"(a0));\n";
    };
    auto emit_load = [&](int s) {
      if (s == 0 && init) os << "        init_regs(R, I, P, W);\n";
      else os << "        load_group_rx<" << (s == 0 ? "true" : "false") << ">(tile, a0, rx, R, I);\n";
      if (s == 0 && fork) emit_fork_scale();
      if (s + 1 == ns && direct)  // the slot is free once every thread of the group has read it
        os << "        fence_proxy_async();\n        mbar_arrive(&empty_bar[slot]);\n";
    };
    // first half of a matrix stage: the rows into TMEM as A
    auto emit_pre = [&](int s) {
      if (s >= ns || msi[s] < 0) return;
      const uint32_t si = dp.stage_begin + (uint32_t)s;
      const bool first = s == first_ms;
      os << "        {  // stage " << si << ": A\n";
      stage_head(si);
      emit_load(s);
      if (first && (restore || f16)) {
        // the tile's norm^2 before the products (compensated warp sums): the restore's
        // reference, and (F16x3) the tile's scale
        os << "        {\n"
           << "          const float2 w = warp_sum2(row_norm2(R, I));\n"
           << "          if (lane == 0) nrm[k & 1][g][0][t >> 5] = w;\n";
        if (f16)
          os << "          group_sync(bar_id, TG);\n"
             << "          sc = tile_scale(nrm[k & 1][g][0]);\n";
        os << "        }\n";
      }
      os << "        matrix_pre<" << (f16 ? "true" : "false") << ", " << (f16 && first ? "true" : "false")
         << ">(R, I, sc, tg, tg + ACOLS, &a_full[g]);\n"
         << "        }\n";
    };
    // second half (or a whole stage without products): D back, the ops, the store
    auto emit_post = [&](int s) {
      const uint32_t si = dp.stage_begin + (uint32_t)s;
      const svp::DevStage &st = P.stages[si];
      const bool last_stage = s + 1 == ns;
      os << "        {  // stage " << si << (msi[s] >= 0 ? ": D" : "") << "\n";
      stage_head(si);
      os << "        int ph = 0;\n        bool zero = false;\n";
      if (msi[s] >= 0)
        os << "        okm &= matrix_post<" << (f16 ? "true" : "false")
           << ">(R, I, tg + 2 * ACOLS, &d_full[g], (uint32_t)((k * NMS + " << msi[s] << ") & 1));\n";
      else
        emit_load(s);
      emit_stage_ops(os, P, st, &pending);
      emit_stage_end(os, &pending, last_stage);
      if (last_stage && f16)  // back from the tile's scale (exact)
        os << "        scale_all(R, I, inv_pow2(sc));\n";
      if (last_stage && restore) {
        // every gate of a PF_UNITARY pass acts inside the tile, so the tile keeps its
        // norm: the products' truncating fp32 accumulation (~0.3 ulp of every output per
        // stage) is undone by scaling the tile to its norm before them, stochastically
        // rounded
        os << "        {  // the tile's norm restored\n"
           << "          const float2 w = warp_sum2(row_norm2(R, I));\n"
           << "          if (lane == 0) nrm[k & 1][g][1][t >> 5] = w;\n"
           << "          group_sync(bar_id, TG);\n"
           << "          const float delta = restore_delta(nrm[k & 1][g][0], nrm[k & 1][g][1]);\n"
           << "          const uint32_t seed = (uint32_t)tile_id * 0x85EBCA6Bu + (uint32_t)(tile_id >> 32) * 0xC2B2AE35u +\n"
           << "                                " << (uint32_t)pass * 0x27D4EB2Fu << "u + (uint32_t)t * 0x165667B1u;\n"
           << "          scale_row_sr(R, I, delta, seed);\n"
           << "        }\n";
      }
      if (!last_stage) {
        os << "        store_group_rx(tile, a0, rx, R, I);\n"
           << "        if (group_any(bar_id, TG, !okm)) { if (t == 0) atomicExch(plan.err, 5); break; }\n"
           << "        }\n";
        return;
      }
      os << "        if (!okm) atomicExch(plan.err, 5);\n";
      if (last) {  // the norm sums, from the registers
        os << "        {\n          float s2 = 0.f, s4 = 0.f;\n"
           << "#pragma unroll\n          for (int p = 0; p < kP; ++p) {\n"
           << "            const float p0 = fmaf(R[p].x, R[p].x, I[p].x * I[p].x), p1 = fmaf(R[p].y, R[p].y, I[p].y * I[p].y);\n"
           << "            s2 += p0 + p1;\n            s4 = fmaf(p0, p0, fmaf(p1, p1, s4));\n"
           << "          }\n          a2 += (double)s2;\n          a4 += (double)s4;\n        }\n";
      }
      if (!direct) {
        os << "        store_group_rx<true>(tile, a0, rx, R, I);\n"
           << "        fence_proxy_async();\n        mbar_arrive(&done_bar[slot]);\n        }\n";
        return;
      }
      os << "        const unsigned long long base = " << tile_base_expr(P, dp) << ";\n"
         << "        const unsigned long long gb = base + (" << group_expr(P, si, "t", true) << ");\n"
         << "        const unsigned long long go[" << (1 << kpr) << "] = {";
      for (int p = 0; p < (1 << kpr); ++p) {
        uint64_t off = 0;
        for (int j = 0; j < kpr; ++j)
          if ((p >> j) & 1) off ^= P.gtab[(size_t)svp::kGroupEntries * si + svp::kRegEntry + j].G;
        os << (p ? ", " : "") << off << "ull";
      }
      os << "};\n"
         << "#pragma unroll\n        for (int p = 0; p < kP; ++p)\n"
         << "          *reinterpret_cast<float4 *>(psi + gb + go[p]) = make_float4(R[p].x, I[p].x, R[p].y, I[p].y);\n"
         << "        }\n";
    };
    os << "      const bool ok = mbar_wait(&full_bar[slot], (uint32_t)((i / S) & 1), kWaitNs);\n"
       << "      if (group_any(bar_id, TG, !ok)) { if (t == 0) atomicExch(plan.err, 3); break; }\n";
    emit_pre(0);
    for (int s = 0; s < ns; ++s) {
      emit_post(s);
      emit_pre(s + 1);
    }
    os << "    }\n  }\n";
  } else {
    os << "  } else {\n"
       << "    // group g takes tiles g, g + G, ...: tile i in slot i mod S (S a multiple of G,\n"
       << "    // so the group's slots g, g + G, ... are only ever its own)\n"
       << "    const int g = tid / TG, t = tid % TG;\n"
       << "    const int bar_id = 1 + g;\n"
       << "    for (unsigned long long i = g;; i += G) {\n"
       << "      " << this_tile
       << "      const int slot = (int)(i % S);\n"
       << "      const bool ok = mbar_wait(&full_bar[slot], (uint32_t)((i / S) & 1), kWaitNs);\n"
       << "      if (group_any(bar_id, TG, !ok)) { if (t == 0) atomicExch(plan.err, 3); break; }\n"
       << "      float4 *tile = reinterpret_cast<float4 *>(smem + slot * TILE_BYTES);\n"
       << "      (void)tile;\n"
       << "      const unsigned long long base = " << tile_base_expr(P, dp) << ";\n"
       << "      (void)base;\n"
       << "      const uint32_t W = ((uint32_t)tile_id << " << (m - 1 - kpr) << ") | (uint32_t)t;\n"
       << "      (void)W;\n";
    if (inner) os << "      const unsigned long long other_base = " << tile_base_expr(P, dp, true) << ";\n";
    int pending = 0;
    const int ns = dp.stage_count;
    for (int s = 0; s < ns; ++s) {
      const uint32_t si = dp.stage_begin + (uint32_t)s;
      const svp::DevStage &st = P.stages[si];
      const bool last_stage = s + 1 == ns;
      os << "      {  // stage " << si << "\n"
         << "      const uint32_t rx[" << kpr << "] = {";
      for (int j = 0; j < kpr; ++j)
        os << (j ? ", " : "") << hex32(P.gtab[(size_t)svp::kGroupEntries * si + svp::kRegEntry + j].L);
      os << "};\n      Regs R, I;\n      int ph = 0;\n      bool zero = false;\n"
         << "      const uint32_t a0 = " << group_expr(P, si, "t", false) << ";\n";
      if (s == 0 && init) {
        os << "      init_regs(R, I, P, W);\n";
      } else if (s == 0 && masked) {
        // zero where a tile bit outside the support is not x's
        uint32_t gm = 0, pm = 0;
        for (int i = 0; i < m - 1 - kpr; ++i) gm |= (uint32_t)!((U >> dp.tq[st.nonr[i]]) & 1ull) << i;
        for (int j = 0; j < kpr; ++j) pm |= (uint32_t)!((U >> dp.tq[st.rbit[j]]) & 1ull) << j;
        os << "      const bool mine = ((uint32_t)t & " << hex32(gm) << ") == ba.group;\n";
        if (U == 0) {  // |x> itself
          os << "#pragma unroll\n      for (int p = 0; p < kP; ++p) {\n"
             << "        const bool hit = mine && (ba.regs & 255u) == (uint32_t)p;\n"
             << "        R[p] = f2(hit && !(ba.regs & 256u) ? 1.f : 0.f, hit && (ba.regs & 256u) ? 1.f : 0.f);\n"
             << "        I[p] = f2(0.f, 0.f);\n      }\n";
        } else {
          os << "      {\n      const unsigned long long g0 = base + (" << group_expr(P, si, "t", true) << ");\n"
             << "      const unsigned long long o0[" << (1 << kpr) << "] = {";
          for (int p = 0; p < (1 << kpr); ++p) {
            uint64_t off = 0;
            for (int j = 0; j < kpr; ++j)
              if ((p >> j) & 1) off ^= P.gtab[(size_t)svp::kGroupEntries * si + svp::kRegEntry + j].G;
            os << (p ? ", " : "") << placed(P, off) << "ull";
          }
          os << "};\n#pragma unroll\n      for (int p = 0; p < kP; ++p) {\n"
             << "        float4 x = make_float4(0.f, 0.f, 0.f, 0.f);\n"
             << "        if (mine && ((uint32_t)p & " << hex32(pm) << ") == ba.regs)\n"
             << "          x = __ldcg(reinterpret_cast<const float4 *>(psi + g0 + o0[p]));\n"
             << "        R[p] = f2(x.x, x.z);\n        I[p] = f2(x.y, x.w);\n      }\n      }\n";
        }
      } else os << "      load_group_rx<" << (s == 0 ? "true" : "false") << ">(tile, a0, rx, R, I);\n";
      if (s == 0 && fork) emit_fork_scale();
      if (last_stage && direct)  // the slot is free once every thread of the group has read it
        os << "      fence_proxy_async();\n      mbar_arrive(&empty_bar[slot]);\n";
      emit_stage_ops(os, P, st, &pending, true);
      emit_stage_end(os, &pending, last_stage);
      if (!last_stage) {
        os << "      store_group_rx(tile, a0, rx, R, I);\n"
           << "      group_sync(bar_id, TG);\n      }\n";
        continue;
      }
      if (last && !inner) {  // the norm sums, from the registers
        os << "      {\n        float s2 = 0.f, s4 = 0.f;\n"
           << "#pragma unroll\n        for (int p = 0; p < kP; ++p) {\n"
           << "          const float p0 = fmaf(R[p].x, R[p].x, I[p].x * I[p].x), p1 = fmaf(R[p].y, R[p].y, I[p].y * I[p].y);\n"
           << "          s2 += p0 + p1;\n          s4 = fmaf(p0, p0, fmaf(p1, p1, s4));\n"
           << "        }\n        a2 += (double)s2;\n        a4 += (double)s4;\n      }\n";
      }
      if (!direct) {
        // back into the slot in memory order; the storer warp writes it out
        os << "      store_group_rx<true>(tile, a0, rx, R, I);\n"
           << "      fence_proxy_async();\n      mbar_arrive(&done_bar[slot]);\n      }\n";
        continue;
      }
      // straight from registers to HBM (pair p at its global index)
      os << "      const unsigned long long gb = " << (inner ? "other_base" : "base") << " + ("
         << group_expr(P, si, "t", true, inner) << ");\n"
         << "      const unsigned long long go[" << (1 << kpr) << "] = {";
      for (int p = 0; p < (1 << kpr); ++p) {
        uint64_t off = 0;
        for (int j = 0; j < kpr; ++j)
          if ((p >> j) & 1) off ^= P.gtab[(size_t)svp::kGroupEntries * si + svp::kRegEntry + j].G;
        os << (p ? ", " : "") << (inner ? off : placed(P, off)) << "ull";
      }
      os << "};\n";
      if (inner) {
        // <this state | other> over the group instead of storing it
        os << "      float sr = 0.f, sim = 0.f;\n"
           << "#pragma unroll\n      for (int p = 0; p < kP; ++p) {\n"
           << "        const float4 y = *reinterpret_cast<const float4 *>(other + gb + go[p]);\n"
           << "        sr = fmaf(R[p].x, y.x, fmaf(I[p].x, y.y, sr));\n"
           << "        sr = fmaf(R[p].y, y.z, fmaf(I[p].y, y.w, sr));\n"
           << "        sim = fmaf(R[p].x, y.y, fmaf(-I[p].x, y.x, sim));\n"
           << "        sim = fmaf(R[p].y, y.w, fmaf(-I[p].y, y.z, sim));\n"
           << "      }\n      a2 += (double)sr;\n      a4 += (double)sim;\n";
      } else {
        os << "#pragma unroll\n      for (int p = 0; p < kP; ++p)\n"
           << "        *reinterpret_cast<float4 *>(psi + gb + go[p]) = make_float4(R[p].x, I[p].x, R[p].y, I[p].y);\n";
      }
      os << "      }\n";
    }
    os << "    }\n  }\n";
  }

  if (mma)
    os << "  // tensor memory is freed once every product and every read of it is done\n"
       << "  fence_before();\n  __syncthreads();\n"
       << "  if (tid >= MT0) {\n    fence_after();\n"
       << "    asm volatile(\"tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\" ::\"r\"(tmem));\n  }\n";
  else
    os << "  __syncthreads();\n";
  if (inner) os << "  block_sums_out(a2, a4, sums);\n";
  else if (last) os << "  if (sums) block_sums_out(a2, a4, sums);\n";
  os << "}\n";
  return os.str();
}

std::string pass_source(const svp::Plan &P, int kpr, int pass, bool inner) {
  std::ostringstream os;
  os << "// tile-pass kernel of one pass of a plan\n#define SV_PACK_R " << kpr
     << "\n#include \"tile_pack.cuh\"\nusing namespace svk::tpk;\n";
  {
    const size_t pi = (size_t)pass;
    const svp::DevPass &dp = P.passes[pi];
    const int threads = 1 << (dp.m - 1 - kpr);
    const bool init = (dp.flags & (svp::PF_INIT_UNIFORM | svp::PF_INIT_ZERO)) != 0;
    // resident CTAs per SM: five of 12-qubit tiles (32 KiB, <= 102 registers; measured
    // best: 34q 0.712 s against 0.739 with four and 0.751 with six), two of 13 (64 KiB),
    // one 512-thread CTA of 14
    const int min_ctas = dp.m <= 12 ? 5 : dp.m == 13 ? 2 : 1;
    os << "\nextern \"C\" __global__ void __launch_bounds__(" << threads << ", " << min_ctas << ")\nsv_pass"
       << "(float2 *__restrict__ psi, svk::DevPlanView plan, unsigned long long num_tiles, double *sums,\n"
       << "        const float2 *__restrict__ other) {\n"
       << "  extern __shared__ __align__(16) unsigned char smem_raw[];\n"
       << "  __shared__ svp::DevPass P;\n"
       << "  __shared__ unsigned long long chunk_off[1 << 10];\n"
       << "  const int tid = threadIdx.x;\n"
       << "  if (tid == 0) P = plan.passes[" << pi << "];\n"
       << "  __syncthreads();\n"
       << "  build_chunk_table(P, chunk_off);\n"
       << "  __syncthreads();\n"
       << "  float4 *tile = reinterpret_cast<float4 *>(smem_raw);\n";
    // the last pass can also sum p and p^2 over the state as it stores it (sums: one
    // pair per CTA, or null)
    const bool last = pi + 1 == P.passes.size();
    inner = inner && last;
    if (last) os << "  double a2 = 0.0, a4 = 0.0;\n";
    else os << "  (void)sums;\n";
    if (!inner) os << "  (void)other;\n";
    os << "  for (unsigned long long tile_id = blockIdx.x; tile_id < num_tiles; tile_id += gridDim.x) {\n"
       << "    const unsigned long long base = tile_base(P, tile_id);\n";
    if (!init) {
      os << "    load_tile_async(psi, tile, P, chunk_off, base);\n"
         << "    finish_tile_copy(tile, P);\n"
         << "    __syncthreads();\n";
    } else if (dp.stage_count == 0) {
      os << "    init_tile(tile, P, base);\n    __syncthreads();\n";
    }
    os << "    const uint32_t W = ((uint32_t)tile_id << " << (dp.m - 1 - kpr) << ") | (uint32_t)tid;\n"
       << "    (void)W;\n";
    int pending = 0;
    for (int s = 0; s < dp.stage_count; ++s) {
      const uint32_t si = dp.stage_begin + (uint32_t)s;
      const svp::DevStage &st = P.stages[si];
      os << "    {  // stage " << si << "\n"
         << "      const uint32_t rx[" << kpr << "] = {";
      for (int j = 0; j < kpr; ++j)
        os << (j ? ", " : "") << hex32(P.gtab[(size_t)svp::kGroupEntries * si + svp::kRegEntry + j].L);
      os << "};\n      Regs R, I;\n      int ph = 0;\n      bool zero = false;\n";
      if (s == 0 && init) os << "      init_regs(R, I, P, W);\n";
      else os << "      load_group_rx<" << (s == 0 ? "true" : "false") << ">(tile, " << group_expr(P, si, "tid", false)
              << ", rx, R, I);\n";
      emit_stage_ops(os, P, st, &pending);
      emit_stage_end(os, &pending, s + 1 == dp.stage_count);
      os << "      store_group_rx(tile, " << group_expr(P, si, "tid", false) << ", rx, R, I);\n"
         << "      __syncthreads();\n    }\n";
    }
    if (inner)  // <this state | other>: the tile is not stored
      os << "    inner_tile(other, tile, P, chunk_off, base, a2, a4);\n    __syncthreads();\n  }\n"
         << "  block_sums_out(a2, a4, sums);\n}\n";
    else if (last)
      os << "    if (sums) store_tile_sums(psi, tile, P, chunk_off, base, a2, a4);\n"
         << "    else store_tile(psi, tile, P, chunk_off, base);\n    __syncthreads();\n  }\n"
         << "  if (sums) block_sums_out(a2, a4, sums);\n}\n";
    else
      os << "    store_tile(psi, tile, P, chunk_off, base);\n    __syncthreads();\n  }\n}\n";
  }
  return os.str();
}

namespace {

// NVRTC, opened at first use: the library loads (and runs every plan on the ahead-of-time
// kernels) where it is missing.
struct Nvrtc {
  bool ok = false;
  std::string why;
  decltype(&nvrtcCreateProgram) create = nullptr;
  decltype(&nvrtcCompileProgram) compile = nullptr;
  decltype(&nvrtcGetProgramLogSize) log_size = nullptr;
  decltype(&nvrtcGetProgramLog) log = nullptr;
  decltype(&nvrtcGetCUBINSize) cubin_size = nullptr;
  decltype(&nvrtcGetCUBIN) cubin = nullptr;
  decltype(&nvrtcDestroyProgram) destroy = nullptr;
  decltype(&nvrtcGetErrorString) error = nullptr;
};

const Nvrtc &nvrtc() {
  static Nvrtc N;
  static std::once_flag once;
  std::call_once(once, [] {
    void *h = nullptr;
    for (const char *name : {"libnvrtc.so.13", "libnvrtc.so", "/usr/local/cuda/lib64/libnvrtc.so.13",
                             "/usr/local/cuda/lib64/libnvrtc.so"}) {
      h = dlopen(name, RTLD_NOW | RTLD_LOCAL);
      if (h) break;
    }
    if (!h) { N.why = "libnvrtc not found"; return; }
    N.create = (decltype(N.create))dlsym(h, "nvrtcCreateProgram");
    N.compile = (decltype(N.compile))dlsym(h, "nvrtcCompileProgram");
    N.log_size = (decltype(N.log_size))dlsym(h, "nvrtcGetProgramLogSize");
    N.log = (decltype(N.log))dlsym(h, "nvrtcGetProgramLog");
    N.cubin_size = (decltype(N.cubin_size))dlsym(h, "nvrtcGetCUBINSize");
    N.cubin = (decltype(N.cubin))dlsym(h, "nvrtcGetCUBIN");
    N.destroy = (decltype(N.destroy))dlsym(h, "nvrtcDestroyProgram");
    N.error = (decltype(N.error))dlsym(h, "nvrtcGetErrorString");
    N.ok = N.create && N.compile && N.log_size && N.log && N.cubin_size && N.cubin && N.destroy && N.error;
    if (!N.ok) N.why = "libnvrtc lacks an entry point";
  });
  return N;
}

}  // namespace

bool compile(const std::string &src, const char *arch, std::string *cubin, std::string *log) {
  const Nvrtc &N = nvrtc();
  if (!N.ok) {
    *log = N.why;
    return false;
  }
  nvrtcProgram prog;
  nvrtcResult r = N.create(&prog, src.c_str(), "sv_plan_kernels.cu", kHeaderCount, kHeaderSources, kHeaderNames);
  if (r != NVRTC_SUCCESS) {
    *log = std::string("nvrtcCreateProgram: ") + N.error(r);
    return false;
  }
  const std::string arch_opt = std::string("--gpu-architecture=") + arch;
  const char *opts[] = {arch_opt.c_str(), "-std=c++17", "-default-device"};
  r = N.compile(prog, 3, opts);
  size_t n = 0;
  N.log_size(prog, &n);
  std::string lg(n, '\0');
  if (n) N.log(prog, &lg[0]);
  while (!lg.empty() && lg.back() == '\0') lg.pop_back();
  *log = lg;
  bool ok = r == NVRTC_SUCCESS;
  if (ok) {
    size_t cb = 0;
    ok = N.cubin_size(prog, &cb) == NVRTC_SUCCESS && cb > 0;
    if (ok) {
      cubin->assign(cb, '\0');
      ok = N.cubin(prog, &(*cubin)[0]) == NVRTC_SUCCESS;
    }
  }
  N.destroy(&prog);
  return ok;
}

namespace {

// Driver-API entry points, taken from the runtime (no link-time dependency on libcuda,
// so the library also loads on a machine without a GPU driver).
struct Driver {
  bool ok = false;
  decltype(&cuModuleLoadData) load = nullptr;
  decltype(&cuModuleUnload) unload = nullptr;
  decltype(&cuModuleGetFunction) get_function = nullptr;
  decltype(&cuFuncSetAttribute) set_attribute = nullptr;
  decltype(&cuOccupancyMaxActiveBlocksPerMultiprocessor) occupancy = nullptr;
  decltype(&cuLaunchKernel) launch = nullptr;
  decltype(&cuGetErrorString) error = nullptr;
  decltype(&cuTensorMapEncodeTiled) encode_tiled = nullptr;
};

template <class F>
bool entry(const char *name, F *fn) {
  void *p = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion(name, &p, CUDA_VERSION, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess || !p)
    return false;
  *fn = reinterpret_cast<F>(p);
  return true;
}

const Driver &driver() {
  static Driver D;
  static std::once_flag once;
  std::call_once(once, [] {
    D.ok = entry("cuModuleLoadData", &D.load) && entry("cuModuleUnload", &D.unload) &&
           entry("cuModuleGetFunction", &D.get_function) && entry("cuFuncSetAttribute", &D.set_attribute) &&
           entry("cuOccupancyMaxActiveBlocksPerMultiprocessor", &D.occupancy) &&
           entry("cuLaunchKernel", &D.launch) && entry("cuGetErrorString", &D.error) &&
           entry("cuTensorMapEncodeTiled", &D.encode_tiled);
  });
  return D;
}

}  // namespace

struct Module {
  int kpr = 0;                // register slots of the plan
  std::vector<CUmodule> mod;  // one per pass
  std::vector<CUfunction> fn;
  std::vector<int> per_sm;  // resident CTAs per SM of each pass kernel
  std::vector<bool> configured;
  std::vector<bool> pipe;   // the pass kernel is the pipelined one (pipe_pass_source)
  std::vector<int> threads; // threads of each pipelined pass kernel's CTA
  std::vector<int> slots;   // shared-memory tile slots of each pipelined pass kernel
  std::vector<size_t> extra;  // further dynamic shared memory (the B buffers of matrix stages)
};

namespace {

std::mutex g_mu;
std::map<std::pair<int, uint64_t>, std::unique_ptr<Module>> g_modules;

uint64_t fnv1a(const std::string &s) {
  uint64_t h = 1469598103934665603ull;
  for (unsigned char c : s) h = (h ^ c) * 1099511628211ull;
  return h;
}

// <directory of this library>/jit, or "" when it cannot be made
std::string cache_dir() {
  Dl_info info;
  if (!dladdr(reinterpret_cast<void *>(&fnv1a), &info) || !info.dli_fname) return "";
  std::string path = info.dli_fname;
  const size_t slash = path.rfind('/');
  if (slash == std::string::npos) return "";
  const std::string dir = path.substr(0, slash) + "/jit";
  mkdir(dir.c_str(), 0755);
  struct stat st;
  if (stat(dir.c_str(), &st) != 0 || !S_ISDIR(st.st_mode)) return "";
  return dir;
}

bool read_file(const std::string &path, std::string *out) {
  std::ifstream f(path, std::ios::binary);
  if (!f) return false;
  std::ostringstream ss;
  ss << f.rdbuf();
  *out = ss.str();
  return !out->empty();
}

void write_file(const std::string &path, const std::string &data) {
  const std::string tmp = path + ".tmp" + std::to_string((long long)getpid());
  {
    std::ofstream f(tmp, std::ios::binary);
    if (!f) return;
    f.write(data.data(), (std::streamsize)data.size());
    if (!f) return;
  }
  std::rename(tmp.c_str(), path.c_str());
}

}  // namespace

namespace {

// The texts of the headers that every source includes: part of a cached cubin's key, as the source
// itself does not change with them.
const std::string &headers_key() {
  static const std::string key = [] {
    std::string all;
    for (int i = 0; i < kHeaderCount; ++i) all += std::string(kHeaderNames[i]) + '\n' + kHeaderSources[i];
    return std::to_string(fnv1a(all));
  }();
  return key;
}

// Compile sources to cubins in a pool of one worker per hardware thread; a cubin whose
// key (source, headers, architecture) is in the cache directory is read instead.  ok[i] = 0
// where NVRTC failed.
void compile_sources(const std::vector<std::string> &src, const char *arch, const std::string &cache,
                     std::vector<std::string> *cubins, std::vector<std::string> *logs, std::vector<char> *ok) {
  const size_t ns = src.size();
  cubins->assign(ns, std::string());
  logs->assign(ns, std::string());
  ok->assign(ns, 1);
  std::vector<std::string> file(ns);
  std::vector<size_t> todo;
  for (size_t i = 0; i < ns; ++i) {
    if (!cache.empty()) {
      char name[96];
      std::snprintf(name, sizeof(name), "/%016llx_%s.cubin", (unsigned long long)fnv1a(src[i] + headers_key() + arch), arch);
      file[i] = cache + name;
      if (read_file(file[i], &(*cubins)[i])) continue;
    }
    todo.push_back(i);
  }
  std::atomic<size_t> next(0);
  auto work = [&] {
    for (size_t t; (t = next.fetch_add(1)) < todo.size();) {
      const size_t i = todo[t];
      (*ok)[i] = compile(src[i], arch, &(*cubins)[i], &(*logs)[i]);
      if ((*ok)[i] && !file[i].empty()) write_file(file[i], (*cubins)[i]);
    }
  };
  const size_t hw = std::max<size_t>(1, std::thread::hardware_concurrency());
  std::vector<std::thread> workers;
  for (size_t w = 0; w < std::min(hw, todo.size()); ++w) workers.emplace_back(work);
  for (std::thread &t : workers) t.join();
}

bool device_arch(char *arch, size_t cap, int *dev) {
  if (cudaGetDevice(dev) != cudaSuccess) return false;
  int major = 0, minor = 0;
  cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, *dev);
  cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, *dev);
  std::snprintf(arch, cap, "sm_%d%da", major, minor);
  return true;
}

}  // namespace

bool pass_is_pipelined(const svp::Plan &P, int pass) {
  int g, s;
  return P.layout == 1 && P.passes[(size_t)pass].stage_count > 0 && pass_pipe_shape(P, pass, &g, &s);
}

bool pass_can_fork(const svp::Plan &P, int bits) {
  if (bits < 1 || P.basis || P.passes.empty() || !pass_is_pipelined(P, 0)) return false;
  const svp::DevPass &hp = P.passes[0];
  if ((hp.flags & (svp::PF_INIT_UNIFORM | svp::PF_INIT_ZERO)) || P.n - hp.m < bits) return false;
  for (int i = 0; i < hp.m; ++i)
    if (hp.tq[i] >= P.n - bits) return false;
  return true;
}

std::string any_pass_source(const svp::Plan &P, int kpr, int pass, bool inner) {
  return pass_is_pipelined(P, pass) ? pipe_pass_source(P, kpr, pass, inner) : pass_source(P, kpr, pass, inner);
}

bool compile_plan(const svp::Plan &P, int kpr, const char *arch, std::vector<std::string> *cubins,
                  std::string *log, const std::string &cache) {
  const size_t np = P.passes.size();
  std::vector<std::string> src(np), logs;
  std::vector<char> ok;
  for (size_t pi = 0; pi < np; ++pi) src[pi] = any_pass_source(P, kpr, (int)pi, false);
  compile_sources(src, arch, cache, cubins, &logs, &ok);
  bool all = true;
  log->clear();
  for (size_t pi = 0; pi < np; ++pi) {
    if (!ok[pi]) all = false;
    if (!logs[pi].empty()) *log += "pass " + std::to_string(pi) + ": " + logs[pi];
  }
  return all;
}

bool get_modules(const std::vector<const svp::Plan *> &plans, int kpr, std::vector<const Module *> *out,
                 std::string *err, bool inner) {
  out->assign(plans.size(), nullptr);
  int dev = 0;
  char arch[32];
  if (!device_arch(arch, sizeof(arch), &dev)) { *err = "no current device"; return false; }
  // the modules load into the runtime's context of this device: make sure it exists
  // (nothing else may have touched the device yet, e.g. a batch with a cached tile size)
  if (cudaFree(nullptr) != cudaSuccess) { *err = "cannot initialise the device context"; return false; }
  // sources of every pass of every plan, keyed per plan by their hash
  std::vector<std::vector<std::string>> src(plans.size());
  std::vector<uint64_t> key(plans.size());
  for (size_t i = 0; i < plans.size(); ++i) {
    std::string all;
    for (size_t pi = 0; pi < plans[i]->passes.size(); ++pi) {
      src[i].push_back(any_pass_source(*plans[i], kpr, (int)pi, inner));
      all += src[i].back();
    }
    key[i] = fnv1a(all + arch);
  }
  std::lock_guard<std::mutex> lock(g_mu);
  std::vector<std::string> flat;
  std::vector<size_t> first(plans.size(), 0);
  std::map<uint64_t, size_t> pending;  // key -> plan whose sources are queued
  for (size_t i = 0; i < plans.size(); ++i) {
    auto it = g_modules.find({dev, key[i]});
    if (it != g_modules.end()) {
      (*out)[i] = it->second.get();
      continue;
    }
    if (pending.count(key[i])) continue;
    pending[key[i]] = i;
    first[i] = flat.size();
    flat.insert(flat.end(), src[i].begin(), src[i].end());
  }
  if (pending.empty()) return true;
  const Driver &D = driver();
  if (!D.ok) { *err = "driver entry points unavailable"; return false; }
  std::vector<std::string> cubins, logs;
  std::vector<char> ok;
  compile_sources(flat, arch, cache_dir(), &cubins, &logs, &ok);
  for (size_t j = 0; j < flat.size(); ++j)
    if (!ok[j]) { *err = "NVRTC compile of the plan kernels failed: " + logs[j].substr(0, 2000); return false; }
  for (const auto &kv : pending) {
    const size_t i = kv.second;
    const size_t np = plans[i]->passes.size();
    std::unique_ptr<Module> M(new Module);
    M->kpr = kpr;
    for (size_t pi = 0; pi < np; ++pi) {
      CUmodule mod = nullptr;
      CUfunction f = nullptr;
      CUresult r = D.load(&mod, cubins[first[i] + pi].data());
      if (r == CUDA_SUCCESS) r = D.get_function(&f, mod, "sv_pass");
      if (r != CUDA_SUCCESS) {
        const char *s = nullptr;
        D.error(r, &s);
        *err = std::string("loading a plan kernel: ") + (s ? s : "?");
        if (mod) D.unload(mod);
        for (CUmodule m : M->mod) D.unload(m);
        return false;
      }
      M->mod.push_back(mod);
      M->fn.push_back(f);
    }
    M->per_sm.assign(np, 0);
    M->configured.assign(np, false);
    M->pipe.assign(np, false);
    M->threads.assign(np, 0);
    M->slots.assign(np, 0);
    M->extra.assign(np, 0);
    for (size_t pi = 0; pi < np; ++pi) {
      M->extra[pi] = pass_mma_smem(*plans[i], (int)pi);
      M->pipe[pi] = pass_is_pipelined(*plans[i], (int)pi);
      if (!M->pipe[pi]) continue;
      int g = 0, sl = 0;
      pass_pipe_shape(*plans[i], (int)pi, &g, &sl);
      M->threads[pi] = pipe_threads(*plans[i], kpr, (int)pi, inner);
      M->slots[pi] = sl;
    }
    // Modules stay loaded for the life of the process (handles and batches keep
    // pointers to them for the circuits they replay); a process that runs many
    // different large circuits holds one set of pass kernels per circuit (about 100 KB
    // of device code per pass).
    g_modules[{dev, key[i]}] = std::move(M);
  }
  for (size_t i = 0; i < plans.size(); ++i)
    if (!(*out)[i]) (*out)[i] = g_modules[{dev, key[i]}].get();
  return true;
}

const Module *get_module(const svp::Plan &P, int kpr, std::string *err, bool inner) {
  std::vector<const Module *> out;
  return get_modules({&P}, kpr, &out, err, inner) ? out[0] : nullptr;
}

namespace {

// Threads and dynamic shared memory of one pass kernel's CTA.
void pass_shape(const Module *M, int pass, int m, int *threads, size_t *smem) {
  if (M->pipe[pass]) {
    *threads = M->threads[pass];
    *smem = (size_t)M->slots[pass] * (sizeof(float2) << m) + M->extra[pass] + 1024;  // + 1 KB alignment
  } else {
    *threads = 1 << (m - 1 - M->kpr);
    *smem = sizeof(float2) << m;
  }
}

// Dynamic shared memory limit and resident CTAs per SM of one pass kernel (once).
bool configure_pass(Module *M, int pass, int m) {
  const Driver &D = driver();
  int threads = 0;
  size_t smem = 0;
  pass_shape(M, pass, m, &threads, &smem);
  std::lock_guard<std::mutex> lock(g_mu);
  if (M->configured[pass]) return true;
  CUfunction f = M->fn[pass];
  if (D.set_attribute(f, CU_FUNC_ATTRIBUTE_MAX_DYNAMIC_SHARED_SIZE_BYTES, (int)smem) != CUDA_SUCCESS) return false;
  int q = 0;
  if (D.occupancy(&q, f, threads, smem) != CUDA_SUCCESS) return false;
  M->per_sm[pass] = q < 1 ? 1 : q;
  M->configured[pass] = true;
  return true;
}

}  // namespace

cudaError_t prepare_passes(const Module *Mc, const svp::Plan &P) {
  Module *M = const_cast<Module *>(Mc);
  if (!driver().ok || P.passes.size() != M->fn.size()) return cudaErrorInvalidValue;
  for (size_t p = 0; p < P.passes.size(); ++p)
    if (!configure_pass(M, (int)p, P.passes[p].m)) return cudaErrorLaunchFailure;
  return cudaSuccess;
}

unsigned max_pass_grid() { return (unsigned)svk::device_sm_count() * 32u; }  // <= 32 CTAs per SM

// One pass over `tiles` tiles; more: the last argument of a kernel that takes one (a basis plan's
// BasisArgs, the first tile of a forking pass), else null.
static cudaError_t launch_tiles(const Module *Mc, float2 *psi, int n, const svk::DevPlanView &view, int pass,
                                const svp::DevPass &hp, uint64_t tiles, void *more, cudaStream_t st, double *sums,
                                unsigned *grid_out, const float2 *other) {
  Module *M = const_cast<Module *>(Mc);
  const Driver &D = driver();
  if (!D.ok || pass < 0 || pass >= (int)M->fn.size()) return cudaErrorInvalidValue;
  const int m = hp.m;
  int threads = 0;
  size_t smem = 0;
  pass_shape(M, pass, m, &threads, &smem);
  if (!configure_pass(M, pass, m)) return cudaErrorLaunchFailure;
  CUfunction f = M->fn[pass];
  uint64_t grid = (uint64_t)svk::device_sm_count() * (uint64_t)M->per_sm[pass];
  if (grid > tiles) grid = tiles;
  unsigned long long num_tiles = tiles;
  svk::DevPlanView v = view;
  if (grid_out) *grid_out = (unsigned)grid;
  CUresult r;
  if (M->pipe[pass]) {
    // The state as a 5-d tensor whose 8-row boxes are one tile's copies: dim 0 = the 32
    // floats of 16 amplitudes (qubits 0..3), dims 1..3 = tile qubits tq[4..6] (extent 2,
    // stride 2^q amplitudes), dim 4 = the 128-byte row at which a box starts (stride
    // 128 B).  A box's rows are thus the 8 combinations of tile qubits tq[4..6] above the
    // box's first row; the 128-byte swizzle puts row r's 16-byte chunk c at c ^ r.
    alignas(64) CUtensorMap map;
    const cuuint64_t dims[5] = {32, 2, 2, 2, (cuuint64_t)1 << (n - 4)};
    const cuuint64_t strides[4] = {(cuuint64_t)8 << hp.tq[4], (cuuint64_t)8 << hp.tq[5], (cuuint64_t)8 << hp.tq[6], 128};
    const cuuint32_t box[5] = {32, 2, 2, 2, 1};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    r = D.encode_tiled(&map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 5, psi, dims, strides, box, estr,
                       CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                       CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cudaErrorInvalidValue;
    void *args[] = {&psi, &v, &num_tiles, &sums, &other, &map, more};
    r = D.launch(f, (unsigned)grid, 1, 1, (unsigned)threads, 1, 1, (unsigned)smem, (CUstream)st, args, nullptr);
  } else {
    void *args[] = {&psi, &v, &num_tiles, &sums, &other};
    r = D.launch(f, (unsigned)grid, 1, 1, (unsigned)threads, 1, 1, (unsigned)smem, (CUstream)st, args, nullptr);
  }
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorLaunchFailure;
}

cudaError_t launch_pass(const Module *M, float2 *psi, int n, const svk::DevPlanView &view, int pass,
                        const svp::DevPass &hp, cudaStream_t st, double *sums, unsigned *grid_out,
                        const float2 *other) {
  return launch_tiles(M, psi, n, view, pass, hp, 1ull << (n - hp.m), nullptr, st, sums, grid_out, other);
}

bool last_pass_tiles(const svp::Plan &P, const std::vector<uint64_t> &needed, uint64_t all_of,
                     std::vector<uint64_t> *tiles) {
  const int last = (int)P.passes.size() - 1;
  if (last < 0 || P.basis || (last == 0 && P.fork) || !pass_is_pipelined(P, last)) return false;
  const svp::DevPass &dp = P.passes.back();
  int all = 0;
  for (int i = 0; i < dp.nt; ++i) all += (int)((all_of >> dp.ntq[i]) & 1ull);
  tiles->clear();
  for (uint64_t x : needed) {
    uint64_t t = 0;
    for (int i = 0; i < dp.nt; ++i)
      if (!((all_of >> dp.ntq[i]) & 1ull)) t |= ((x >> dp.ntq[i]) & 1ull) << i;
    tiles->push_back(t);
  }
  std::sort(tiles->begin(), tiles->end());
  tiles->erase(std::unique(tiles->begin(), tiles->end()), tiles->end());
  return !tiles->empty() && (tiles->size() << all) <= (1ull << dp.nt) / 2;
}

cudaError_t launch_listed_pass(const Module *M, float2 *psi, const svk::DevPlanView &view, const svp::Plan &P,
                               const uint64_t *tiles, size_t count, cudaStream_t st) {
  return launch_tiles(M, psi, P.n, view, (int)P.passes.size() - 1, P.passes.back(),
                      (uint64_t)count << __builtin_popcountll(listed_bits(P)), &tiles, st, nullptr, nullptr, nullptr);
}

cudaError_t launch_fork_pass(const Module *M, float2 *psi, const svk::DevPlanView &view, const svp::Plan &P,
                             cudaStream_t st) {
  const svp::DevPass &hp = P.passes[0];
  const uint64_t tiles = 1ull << (P.n - hp.m);
  unsigned long long first = tiles >> P.fork;  // the prefix's own tiles come last
  cudaError_t e = launch_tiles(M, psi, P.n, view, 0, hp, tiles - first, &first, st, nullptr, nullptr, nullptr);
  const uint64_t own = first;
  first = 0;
  if (e == cudaSuccess) e = launch_tiles(M, psi, P.n, view, 0, hp, own, &first, st, nullptr, nullptr, nullptr);
  return e;
}

cudaError_t launch_basis_pass(const Module *M, float2 *psi, const svk::DevPlanView &view, const svp::Plan &P, int pass,
                              uint64_t x, cudaStream_t st, double *sums, unsigned *grid_out, const float2 *other) {
  const svp::DevPass &hp = P.passes[(size_t)pass];
  if (!pass_is_pipelined(P, pass)) return cudaErrorInvalidValue;
  const uint64_t U = support(P, pass);
  svk::BasisArgs ba = {0, 0, 0};
  int vary = 0;  // tile index bits of the support
  for (int i = 0; i < hp.nt; ++i) {
    if ((U >> hp.ntq[i]) & 1ull) ++vary;
    else ba.fixed |= ((x >> hp.ntq[i]) & 1ull) << i;
  }
  const svp::DevStage &s0 = P.stages[hp.stage_begin];
  auto bit = [&](int tile_bit) -> uint32_t {
    const int q = hp.tq[tile_bit];
    return ((U >> q) & 1ull) ? 0u : (uint32_t)((x >> q) & 1ull);
  };
  for (int i = 0; i < hp.m - 1 - M->kpr; ++i) ba.group |= bit(s0.nonr[i]) << i;
  for (int j = 0; j < M->kpr; ++j) ba.regs |= bit(s0.rbit[j]) << j;
  ba.regs |= bit(0) << 8;
  svp::DevPass at = hp;  // the tile's rows as they lie in the compact state
  for (int i = 4; i < 7; ++i) at.tq[i] = (uint8_t)std::max(place(P, hp.tq[i]), 4);
  return launch_tiles(M, psi, basis_state_bits(P), view, pass, at, 1ull << vary, &ba, st, sums, grid_out, other);
}

int basis_state_bits(const svp::Plan &P) {
  return std::max(__builtin_popcountll(support(P, (int)P.passes.size() - 1)), 7);
}

}  // namespace svj
