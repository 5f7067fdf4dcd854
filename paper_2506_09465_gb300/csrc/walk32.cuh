// What the FP32 walks share (sweep_staged.cu, land.cu): the error bounds within which their
// decisions are the FP64 walk's, the queue of the particles left to the FP64 replay, and the
// compensated FP32 tally.
#pragma once

#include <cuda_runtime.h>

#include "layout.h"
#include "staged.h"

namespace iugkp {

// i as a float for 0 <= i < 2^23, placed in the mantissa of 2^23 (no conversion instruction).
__device__ __forceinline__ float small_int_float(int i) { return __int_as_float(0x4B000000 | i) - 8388608.f; }

// ---- FP32 decisions checked against the FP64 walk ----
// The FP32 walk and the FP64 walk follow each particle with the same draws, so their path
// lengths differ by rounding only, and a decision taken in FP32 is the FP64 walk's unless the
// FP32 value lies within a bound of the decision's boundary: a face (the count of faces before
// a candidate along an axis, hence its cell), the first wall (a candidate or an absorption),
// the acceptance ratio. A particle with such a decision is not tallied further: it goes to a
// queue that the FP64 walk replays after the sweep (replay_kernel, adjoint_replay_kernel).
// Path-length bounds, FP32 against FP64:
//  * a face count's quotient u = (D - t) / d, times d: TIE_REL (D + d) + eD, TIE_REL covering
//    the rounding of the direction (sqrtf, sincospif, products), cell size, first-face
//    distance, quotient (__fdividef) and difference, about 2^-19.4 in all, taken as 2^-18;
//    the wall distance tex likewise within TIE_REL tex;
//  * eD bounds |D32 - D64|: per flight TIE_LOG_ABS v tau_maj + TIE_LOG_REL l for the fast
//    logarithm, the FP32 v tau_maj and the product's rounding, plus TIE_SUM D for each
//    addition to D. The logarithm's error over all 2^23 uniforms the walk draws is measured
//    (walk_bounds_kernel) at about a third of its share of this allowance.
// The acceptance ratio in FP32 is within 2^-24 of the FP64 ratio (both below 1).
constexpr float TIE_REL = 0x1p-18f;
constexpr float TIE_LOG_ABS = 0x1p-22f;
constexpr float TIE_LOG_REL = 0x1p-20f;
constexpr float TIE_SUM = 0x1p-23f;
constexpr float TIE_ACC = 0x1p-24f;


// Queues a particle for the FP64 replay: forward index and (candidates tallied << 1) | group.
__device__ __forceinline__ void defer_particle(const StagedArgs& S, unsigned pid, unsigned meta) {
  const unsigned i = atomicAdd(S.defer_n, 1u);
  if (i < S.defer_cap) S.defer[i] = make_uint2(pid, meta);
  else atomicOr(S.err, ERR_DEFER);
}

// Compensated FP32 tally. The atomic returns the value it added to, so the exact rounding
// error of the stored sum is known locally (Knuth's TwoSum, six FP32 operations); that error
// and the low part of the FP64 addend go to the companion word. After n additions the pair
// holds the sum to about n 2^-48 relative. (atom.add.f32 flushes subnormal results to zero:
// an absolute error below 2^-126 per addition, far under the tally scale.)
__device__ __forceinline__ void tally_k32(float2* p, double x) {
  const float xh = __double2float_rn(x);
  const float xl = __double2float_rn(x - (double)xh);
  const float old = atomicAdd(&p->x, xh);
  const float sum = __fadd_rn(old, xh);
  const float bv = __fsub_rn(sum, old);
  const float err = __fadd_rn(__fsub_rn(old, __fsub_rn(sum, bv)), __fsub_rn(xh, bv));
  const float lo = __fadd_rn(err, xl);
  if (lo != 0.f) atomicAdd(&p->y, lo);
}

}  // namespace iugkp
