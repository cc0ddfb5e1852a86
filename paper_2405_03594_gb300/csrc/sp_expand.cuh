// sp_expand.cuh -- expanding a few columns of a chunk row from its mask bits and its packed
// values in shared memory, shared by the kernels that need dense columns.
//
// A thread walks its columns in order: each column costs one predicate-setting AND, one
// predicated shared load and one predicated pointer increment, so a dropped column touches
// no shared memory.  Written in PTX to keep that shape; volatile, so that the loads stay
// before the barrier arrive that gives the ring slot back.
#pragma once

#include "sp_internal.cuh"

namespace sp {

// Columns of mask bits B0, B1 as two bf16 (low half, high half): kept columns take the next
// values of the stream at shared address `pa` (which advances); a dropped column is +0.
template <uint32_t B0, uint32_t B1>
__device__ __forceinline__ uint32_t expand_word_bf16(uint32_t m, uint32_t& pa) {
  uint32_t o;
  asm volatile("{\n\t.reg .pred p0, p1;\n\t.reg .b32 t0, t1, lo, hi;\n\t"
      "and.b32 t0, %2, %3;\n\t"
      "setp.ne.b32 p0, t0, 0;\n\t"
      "and.b32 t1, %2, %4;\n\t"
      "setp.ne.b32 p1, t1, 0;\n\t"
      "mov.b32 lo, 0;\n\t"
      "mov.b32 hi, 0;\n\t"
      "@p0 ld.shared.u16 lo, [%1];\n\t"
      "@p0 add.u32 %1, %1, 2;\n\t"
      "@p1 ld.shared.u16 hi, [%1];\n\t"
      "@p1 add.u32 %1, %1, 2;\n\t"
      "prmt.b32 %0, lo, hi, 0x5410;\n\t}"
      : "=r"(o), "+r"(pa)
      : "r"(m), "n"(B0), "n"(B1));
  return o;
}

// The same for one-byte values: the two columns' bytes in bits 0-7 and 16-23, zero elsewhere.
template <uint32_t B0, uint32_t B1>
__device__ __forceinline__ uint32_t expand_word_u8(uint32_t m, uint32_t& pa) {
  uint32_t o;
  asm volatile("{\n\t.reg .pred p0, p1;\n\t.reg .b32 t0, t1, lo, hi;\n\t"
      "and.b32 t0, %2, %3;\n\t"
      "setp.ne.b32 p0, t0, 0;\n\t"
      "and.b32 t1, %2, %4;\n\t"
      "setp.ne.b32 p1, t1, 0;\n\t"
      "mov.b32 lo, 0;\n\t"
      "mov.b32 hi, 0;\n\t"
      "@p0 ld.shared.u8 lo, [%1];\n\t"
      "@p0 add.u32 %1, %1, 1;\n\t"
      "@p1 ld.shared.u8 hi, [%1];\n\t"
      "@p1 add.u32 %1, %1, 1;\n\t"
      "prmt.b32 %0, lo, hi, 0x5410;\n\t}"
      : "=r"(o), "+r"(pa)
      : "r"(m), "n"(B0), "n"(B1));
  return o;
}

// Two signed bytes (bits 0-7 and 16-23 of w, zero elsewhere) as bf16x2, exactly.  128 plus the
// byte's low seven bits is the bf16 0x4300 | low7, and its sign bit, weight -128, turns the
// 128 = 0x4300 to subtract into 256 = 0x4380: one subtraction of two exact bf16 leaves q.
__device__ __forceinline__ uint32_t sub_bf16x2(uint32_t a, uint32_t b) {
  uint32_t o;
  asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(o) : "r"(a), "r"(b));
  return o;
}
__device__ __forceinline__ uint32_t i8x2_to_bf16x2(uint32_t w) {
  return sub_bf16x2((w & 0x007f007fu) | 0x43004300u, (w & 0x00800080u) | 0x43004300u);
}

}  // namespace sp
