// The gate loop of the interpreting kernels, in PTX.
//
// A stage's gates run on a thread's packed amplitude pairs, which stay in registers from the
// stage's load to its store.  As a C++ switch the loop cost more than the gates (190
// instructions and 8 branches an op by the counters, where a rotation on 32 amplitudes needs 32
// packed ones).  Written as one block of PTX the loop is threaded -- every case ends in an
// indexed branch (brx.idx) to the next op's -- and updates its registers in place.
// Measured on one GB300, us a circuit (the switch over 140 unrolled op cases, the plan read
// from global memory / the same as a switch over fewer cases, the plan in shared memory /
// this loop): 12 qubits depth 16 30 / 22 / 18, 16 qubits depth 10 39 / 28 / 21, 23 qubits
// depth 16 350 / 200 / 164.  At 23 qubits an op takes 65 instructions (190 at first), the
// issue slots are 55 % and the FMA pipe 44 % busy; what is left is instruction fetch and the
// branches with 16 warps an SM to cover them.
#pragma once

#include <cuda_runtime.h>

#include "interp_dev.h"

namespace svk {
namespace itp {

// A pair's two floats in one 64-bit register (low word: pack bit 0).
typedef unsigned long long P2;
// RK register slots besides the pack bit: 2^RK pairs a thread
template <int RK>
using PRegs = P2[1 << RK];

// ---- text of the loop ------------------------------------------------------------------------
// Registers r<p>, i<p>: re and im of pair p.  An op is two words (IGate): w (code in the low
// bits, sign and rounding flags on top) and par.  w1, par1: the next op, read ahead.

// (pairs of elements that differ in slot J, by register width)
#define SVG_PAIRS_4_0(M) M(0, 1) M(2, 3) M(4, 5) M(6, 7) M(8, 9) M(10, 11) M(12, 13) M(14, 15)
#define SVG_PAIRS_4_1(M) M(0, 2) M(1, 3) M(4, 6) M(5, 7) M(8, 10) M(9, 11) M(12, 14) M(13, 15)
#define SVG_PAIRS_4_2(M) M(0, 4) M(1, 5) M(2, 6) M(3, 7) M(8, 12) M(9, 13) M(10, 14) M(11, 15)
#define SVG_PAIRS_4_3(M) M(0, 8) M(1, 9) M(2, 10) M(3, 11) M(4, 12) M(5, 13) M(6, 14) M(7, 15)
#define SVG_PAIRS_2_0(M) M(0, 1) M(2, 3)
#define SVG_PAIRS_2_1(M) M(0, 2) M(1, 3)
// (all pairs)
#define SVG_ALL_2(M) M(0) M(1) M(2) M(3)
#define SVG_ALL_4(M) \
  SVG_ALL_2(M) M(4) M(5) M(6) M(7) M(8) M(9) M(10) M(11) M(12) M(13) M(14) M(15)

// The next op: its words were read ahead; read the one after it.
#define SVG_NEXT                                  \
  "mov.b32 w, w1; mov.b32 par, par1;\n"           \
  "ld.shared.v2.b32 {w1, par1}, [at];\n"          \
  "add.u32 at, at, 8; and.b32 c, w, 63;\n"        \
  "brx.idx c, TS;\n"
// s2 = (s, s), n2 = (-s, -s): s = -1 where w's top bit is set
#define SVG_SIGN_OPERANDS                                             \
  "and.b32 t, w, 0x80000000; or.b32 t, t, 0x3f800000;\n"              \
  "xor.b32 u, t, 0x80000000; mov.b64 s2, {t, t}; mov.b64 n2, {u, u};\n" \
  "mov.b32 s, t; mov.b32 n, u;\n"
// q: the sign of the op's slot-1 elements is -1
#define SVG_PARITY "and.b32 t, W, par; popc.b32 t, t; and.b32 t, t, 1; setp.ne.u32 q, t, 0;\n"

#define SVG_NEG_HI(x, y) "mul.rn.f32x2 r" #y ", r" #y ", m1; mul.rn.f32x2 i" #y ", i" #y ", m1;\n"
#define SVG_NEG_P(p) "mul.rn.f32x2 r" #p ", r" #p ", pm; mul.rn.f32x2 i" #p ", i" #p ", pm;\n"
#define SVG_IM(x, y)                                    \
  "fma.rn.f32x2 a, i" #y ", s2, r" #x ";\n"             \
  "fma.rn.f32x2 b, r" #y ", n2, i" #x ";\n"             \
  "fma.rn.f32x2 i" #y ", r" #x ", n2, i" #y ";\n"       \
  "fma.rn.f32x2 r" #y ", i" #x ", s2, r" #y ";\n"       \
  "mov.b64 r" #x ", a; mov.b64 i" #x ", b;\n"
#define SVG_RE(x, y)                                    \
  "fma.rn.f32x2 a, r" #y ", n2, r" #x ";\n"             \
  "fma.rn.f32x2 b, i" #y ", n2, i" #x ";\n"             \
  "fma.rn.f32x2 r" #y ", r" #x ", s2, r" #y ";\n"       \
  "fma.rn.f32x2 i" #y ", i" #x ", s2, i" #y ";\n"       \
  "mov.b64 r" #x ", a; mov.b64 i" #x ", b;\n"
#define SVG_H(x, y)                                     \
  "fma.rn.f32x2 a, r" #y ", p1, r" #x ";\n"             \
  "fma.rn.f32x2 b, i" #y ", p1, i" #x ";\n"             \
  "fma.rn.f32x2 r" #y ", r" #y ", m1, r" #x ";\n"       \
  "fma.rn.f32x2 i" #y ", i" #y ", m1, i" #x ";\n"       \
  "mov.b64 r" #x ", a; mov.b64 i" #x ", b;\n"
#define SVG_T(x, y)                                     \
  "fma.rn.f32x2 a, i" #y ", n2, r" #y ";\n"             \
  "fma.rn.f32x2 b, r" #y ", s2, i" #y ";\n"             \
  "mul.rn.f32x2 r" #y ", a, c2; mul.rn.f32x2 i" #y ", b, c2;\n"
// the same inside a pair (x, x' = its low and high halves)
#define SVG_UNPACK(p) "mov.b64 {e, f}, r" #p "; mov.b64 {g, h}, i" #p ";\n"
#define SVG_PACK(p) "mov.b64 r" #p ", {j, k}; mov.b64 i" #p ", {l, m};\n"
#define SVG_IM_P(p)                                                              \
  SVG_UNPACK(p)                                                                  \
  "fma.rn.f32 j, h, s, e; fma.rn.f32 l, f, n, g; fma.rn.f32 k, g, s, f; fma.rn.f32 m, e, n, h;\n" SVG_PACK(p)
#define SVG_RE_P(p)                                                              \
  SVG_UNPACK(p)                                                                  \
  "fma.rn.f32 j, f, n, e; fma.rn.f32 l, h, n, g; fma.rn.f32 k, e, s, f; fma.rn.f32 m, g, s, h;\n" SVG_PACK(p)
#define SVG_H_P(p)                                                               \
  SVG_UNPACK(p) "add.rn.f32 j, e, f; sub.rn.f32 k, e, f; add.rn.f32 l, g, h; sub.rn.f32 m, g, h;\n" SVG_PACK(p)
#define SVG_T_P(p)                                                               \
  SVG_UNPACK(p)                                                                  \
  "fma.rn.f32 k, h, n, f; fma.rn.f32 m, f, s, h; mul.rn.f32 k, k, cc; mul.rn.f32 m, m, cc;\n" \
  "mov.b64 r" #p ", {e, k}; mov.b64 i" #p ", {g, m};\n"
#define SVG_RS(p)                                                                \
  "mul.rn.f32x2 a, r" #p ", lo; mul.rn.f32x2 b, i" #p ", lo;\n"                  \
  "fma.rn.f32x2 r" #p ", r" #p ", hi, a; fma.rn.f32x2 i" #p ", i" #p ", hi, b;\n"

// the cases of one register slot / of the pack bit
#define SVG_SLOT(J, PAIRS)                                                                  \
  "IM" #J ": " SVG_SIGN_OPERANDS SVG_PARITY "@!q bra IMX" #J ";\n" PAIRS(SVG_NEG_HI)         \
  "IMX" #J ": " PAIRS(SVG_IM) SVG_NEXT                                                      \
  "RE" #J ": " SVG_SIGN_OPERANDS SVG_PARITY "@!q bra REX" #J ";\n" PAIRS(SVG_NEG_HI)         \
  "REX" #J ": " PAIRS(SVG_RE) SVG_NEXT                                                      \
  "H" #J ": " PAIRS(SVG_H) SVG_NEXT                                                         \
  "T" #J ": " SVG_T_OPERANDS PAIRS(SVG_T) SVG_NEXT                                          \
  "S" #J ": " SVG_PARITY "@!q bra SX" #J ";\n" PAIRS(SVG_NEG_HI) "SX" #J ": " SVG_NEXT       \
  "CP" #J ": " PAIRS(SVG_NEG_P2) SVG_NEXT
#define SVG_NEG_P2(x, y) SVG_NEG_P(y)
#define SVG_T_OPERANDS                                                                      \
  SVG_SIGN_OPERANDS                                                                         \
  "and.b32 t, w, 0x40000000; setp.ne.u32 q, t, 0; selp.f32 cc, 0f3F3504F4, 0f3F3504F3, q;\n" \
  "mov.b64 c2, {cc, cc};\n"
#define SVG_PACKSLOT(ALL)                                                                   \
  "IM4: " SVG_SIGN_OPERANDS SVG_PARITY "@!q bra IMX4;\n" ALL(SVG_NEG_P) "IMX4: " ALL(SVG_IM_P) SVG_NEXT \
  "RE4: " SVG_SIGN_OPERANDS SVG_PARITY "@!q bra REX4;\n" ALL(SVG_NEG_P) "REX4: " ALL(SVG_RE_P) SVG_NEXT \
  "H4: " ALL(SVG_H_P) SVG_NEXT                                                              \
  "T4: " SVG_T_OPERANDS ALL(SVG_T_P) SVG_NEXT                                               \
  "S4: " SVG_PARITY "@!q bra SX4;\n" ALL(SVG_NEG_P) "SX4: " SVG_NEXT                         \
  "RS: " ALL(SVG_RS) SVG_NEXT
// CZ of two register slots: the elements where both are 1
#define SVG_NEG(p) "mul.rn.f32x2 r" #p ", r" #p ", m1; mul.rn.f32x2 i" #p ", i" #p ", m1;\n"
#define SVG_CZ(N, A, B, C, D) "C" #N ": " SVG_NEG(A) SVG_NEG(B) SVG_NEG(C) SVG_NEG(D) SVG_NEXT

#define SVG_HEAD                                                                 \
  "{\n .reg .pred q;\n .reg .b32 w, par, w1, par1, at, W, c, t, u;\n"            \
  " .reg .b64 s2, n2, c2, a, b, m1, p1, pm, hi, lo;\n"                           \
  " .reg .f32 s, n, cc, e, f, g, h, j, k, l, m;\n"
#define SVG_DECL(p) " .reg .b64 r" #p ", i" #p ";\n"
#define SVG_CONSTANTS                                                            \
  "mov.b32 t, 0xbf800000; mov.b32 u, 0x3f800000;\n"                              \
  "mov.b64 m1, {t, t}; mov.b64 p1, {u, u}; mov.b64 pm, {u, t};\n"                \
  "mov.b32 t, 0x3f3504f3; mov.b32 u, 0x324fe77a;\n"                              \
  "mov.b64 hi, {t, t}; mov.b64 lo, {u, u};\n"
// the first two ops, then the first dispatch
#define SVG_START                                                                \
  "ld.shared.v2.b32 {w, par}, [at]; ld.shared.v2.b32 {w1, par1}, [at+8];\n"      \
  "add.u32 at, at, 16; and.b32 c, w, 63;\n brx.idx c, TS;\n"

// Ops from shared-memory address `at` (two words each) to the one with code G_END, on a
// thread whose condition word is W (its top bit set: the constant bit of the parities).
// The op after the end is read, never used.
template <int RK>
__device__ __forceinline__ void run_gates(PRegs<RK> &R, PRegs<RK> &I, uint32_t at, uint32_t W);

#define SVG_IN(p, a, b) "mov.b64 r" #p ", %" #a "; mov.b64 i" #p ", %" #b ";\n"
#define SVG_OUT(p, a, b) "mov.b64 %" #a ", r" #p "; mov.b64 %" #b ", i" #p ";\n"

#define SVG_IO_2(M) M(0, 0, 4) M(1, 1, 5) M(2, 2, 6) M(3, 3, 7)
template <>
__device__ __forceinline__ void run_gates<2>(PRegs<2> &R, PRegs<2> &I, uint32_t at, uint32_t W) {
  asm volatile(
      SVG_HEAD SVG_ALL_2(SVG_DECL) SVG_IO_2(SVG_IN) "mov.b32 at, %8; mov.b32 W, %9;\n" SVG_CONSTANTS
      "TS: .branchtargets IM0, IM1, IM0, IM0, IM4, RE0, RE1, RE0, RE0, RE4, H0, H1, H0, H0, H4, T0, T1, T0, T0, T4,"
      " S0, S1, S0, S0, S4, C0, C0, C0, C0, C0, C0, CP0, CP1, CP0, CP0, RS, END;\n" SVG_START
      SVG_SLOT(0, SVG_PAIRS_2_0) SVG_SLOT(1, SVG_PAIRS_2_1) SVG_PACKSLOT(SVG_ALL_2)
      "C0: " SVG_NEG(3) SVG_NEXT
      "END:\n" SVG_IO_2(SVG_OUT) "}\n"
      : "+l"(R[0]), "+l"(R[1]), "+l"(R[2]), "+l"(R[3]), "+l"(I[0]), "+l"(I[1]), "+l"(I[2]), "+l"(I[3])
      : "r"(at), "r"(W)
      : "memory");
}
#undef SVG_IO_2

#define SVG_IO_4(M)                                                                                          \
  M(0, 0, 16) M(1, 1, 17) M(2, 2, 18) M(3, 3, 19) M(4, 4, 20) M(5, 5, 21) M(6, 6, 22) M(7, 7, 23) M(8, 8, 24) \
  M(9, 9, 25) M(10, 10, 26) M(11, 11, 27) M(12, 12, 28) M(13, 13, 29) M(14, 14, 30) M(15, 15, 31)
template <>
__device__ __forceinline__ void run_gates<4>(PRegs<4> &R, PRegs<4> &I, uint32_t at, uint32_t W) {
  asm volatile(
      SVG_HEAD SVG_ALL_4(SVG_DECL) SVG_IO_4(SVG_IN) "mov.b32 at, %32; mov.b32 W, %33;\n" SVG_CONSTANTS
      "TS: .branchtargets IM0, IM1, IM2, IM3, IM4, RE0, RE1, RE2, RE3, RE4, H0, H1, H2, H3, H4, T0, T1, T2, T3, T4,"
      " S0, S1, S2, S3, S4, C0, C1, C2, C3, C4, C5, CP0, CP1, CP2, CP3, RS, END;\n" SVG_START
      SVG_SLOT(0, SVG_PAIRS_4_0) SVG_SLOT(1, SVG_PAIRS_4_1) SVG_SLOT(2, SVG_PAIRS_4_2) SVG_SLOT(3, SVG_PAIRS_4_3)
      SVG_PACKSLOT(SVG_ALL_4)
      SVG_CZ(0, 3, 7, 11, 15) SVG_CZ(1, 5, 7, 13, 15) SVG_CZ(2, 9, 11, 13, 15) SVG_CZ(3, 6, 7, 14, 15)
      SVG_CZ(4, 10, 11, 14, 15) SVG_CZ(5, 12, 13, 14, 15)
      "END:\n" SVG_IO_4(SVG_OUT) "}\n"
      : "+l"(R[0]), "+l"(R[1]), "+l"(R[2]), "+l"(R[3]), "+l"(R[4]), "+l"(R[5]), "+l"(R[6]), "+l"(R[7]), "+l"(R[8]),
        "+l"(R[9]), "+l"(R[10]), "+l"(R[11]), "+l"(R[12]), "+l"(R[13]), "+l"(R[14]), "+l"(R[15]), "+l"(I[0]),
        "+l"(I[1]), "+l"(I[2]), "+l"(I[3]), "+l"(I[4]), "+l"(I[5]), "+l"(I[6]), "+l"(I[7]), "+l"(I[8]), "+l"(I[9]),
        "+l"(I[10]), "+l"(I[11]), "+l"(I[12]), "+l"(I[13]), "+l"(I[14]), "+l"(I[15])
      : "r"(at), "r"(W)
      : "memory");
}
#undef SVG_IO_4

}  // namespace itp
}  // namespace svk
