// The Jacobi preconditioner z = v / (w - i eta + m_nu) in FP32, formed wherever z is used (operand preparation,
// combine pass, correction) instead of being stored. The sum w + m_nu can cancel near a pole: both terms are
// held as pairs of FP32 numbers, so that it is rounded once, as its FP64 value would be. (internal)
#pragma once
#include "gfcc_internal.cuh"

namespace gfcc {

// What a column (its shift) and a row (diagonal entries) bring, converted once: an FP64 conversion or addition
// holds a scheduler for 75 clocks on this GPU, and the kernels that use these would issue one per thread or row.
using ShiftF = float4;   // (w = x + y, -eta = z)
using RowF = float4;     // (m_nu = x + y, the Fock diagonal z)
__device__ __forceinline__ float2 precond_f32(float2 v, const RowF& md, const ShiftF& s) {
  const float a = __fadd_rn(s.x, md.x), bb = __fsub_rn(a, s.x);
  const float e = __fadd_rn(__fsub_rn(s.x, __fsub_rn(a, bb)), __fsub_rn(md.x, bb));   // a + e = s.x + md.x
  const float dr = a + (e + (s.y + md.y)), di = s.z;
  const float inv = 1.0f / (dr * dr + di * di);
  return make_float2((v.x * dr + v.y * di) * inv, (v.y * dr - v.x * di) * inv);
}

}  // namespace gfcc
