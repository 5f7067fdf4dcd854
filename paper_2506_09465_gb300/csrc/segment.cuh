// The straight segment of a particle in the FP32 sweeps (sweep_staged.cu, sweep_chain.cu): the faces
// it crosses per axis, the wall it reaches, and the outcome of a candidate on it, each with the
// bound within which the decision is the FP64 walk's (walk32.cuh).
#pragma once

#include <cuda_runtime.h>

#include "device.cuh"
#include "internal.h"
#include "staged.h"
#include "walk32.cuh"

namespace iugkp {

struct LCounts {
  unsigned v[CNT_N];  // per thread and launch: far below 2^32
};

__device__ __forceinline__ void flush_lcounts(LCounts& c, unsigned long long* out) {
  if (!out) return;
#pragma unroll
  for (int k = 0; k < CNT_N; ++k) {
    unsigned long long x = c.v[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0 && x) atomicAdd(&out[k], x);
  }
}

// Register-resident path state. The direction does not change at null collisions, so the
// path from emission to the end (real collision or wall) is one straight segment: i_a is
// the emission cell, t_a the path length at which the first face normal to axis a is
// reached, d_a the path length per cell along a (+inf when s_a = 0), so the k-th face along
// a is reached at t_a + k d_a. D: path length of the current candidate collision;
// tex: path length at which the segment leaves the domain.
struct PW {
  int i0, i1, i2;
  int s0, s1, s2;
  float t0, t1, t2;
  float d0, d1, d2;
  float D, tex;
};

__device__ __forceinline__ void axis_init(float s, float xi, float h, float& t, float& d, int& st) {
  const float as = fabsf(s);
  st = s > 0.f ? 1 : -1;
  d = __fdividef(h, as);  // +inf when s = 0
  t = (s > 0.f ? 1.f - xi : xi) * d;
}

// ceil(max(u, 0)) for u < 2^23 without a float-to-integer conversion: adding 2^23 with
// rounding upwards lands on 2^23 + ceil(u), whose bits minus those of 2^23 are the count.
__device__ __forceinline__ int ceil_count(float u) {
  return __float_as_int(__fadd_ru(fmaxf(u, 0.f), 8388608.f)) - 0x4B000000;
}

// Faces normal to one axis reached before path length L: #{k >= 0 : t + k d < L}.
__device__ __forceinline__ int faces_before(float L, float t, float d) {
  return L > t ? ceil_count(__fdividef(L - t, d)) : 0;
}

// Faces up to and including the wall along one axis, and the path length of the wall face.
__device__ __forceinline__ int faces_to_wall(int i, int s, int n) { return s > 0 ? n - i : i + 1; }
__device__ __forceinline__ float axis_exit(int i, int s, int n, float t, float d) {
  const int m = faces_to_wall(i, s, n);
  return m > 1 ? fmaf(small_int_float(m - 1), d, t) : t;
}

__device__ __forceinline__ int clampi(int v, int n) { return min(max(v, 0), n - 1); }

// Tie bits of one axis for the count n = faces_before(D, t, d): bit sh when D lies within the
// bound (base = TIE_REL D + eD, plus TIE_REL d) below a face, so that the FP64 walk may count
// one face more; bit sh + 1 when within it above one (one fewer). None when d = inf (NaN).
__device__ __forceinline__ unsigned tie_bits(float D, float t, float d, float base, int n, int sh) {
  const float u = __fdividef(D - t, d);
  const float fr = small_int_float(n) - u;  // up to the next face, in cells: [0, 1]
  const float tol = fmaf(TIE_REL, d, base);
  if (fr * d <= tol) return 1u << sh;
  if ((1.f - fr) * d <= tol && n > 0) return 2u << sh;
  return 0u;
}

// faces_before, and in `near` whether D lies within the bound of a face of this axis (either
// side; the direction is not needed when every candidate is real).
__device__ __forceinline__ int count_near(float D, float t, float d, float base, bool& near) {
  const float u = __fdividef(D - t, d);
  const float c = __fadd_ru(fmaxf(u, 0.f), 8388608.f);  // 2^23 + ceil(max(u, 0))
  const float fr = (c - 8388608.f) - u;
  near |= fminf(fr, 1.f - fr) * d <= fmaf(TIE_REL, d, base);
  return __float_as_int(c) - 0x4B000000;
}

// Axis a's bit of `hit` when the count one more than n reaches the wall (m faces to it).
__device__ __forceinline__ unsigned tie_hits_wall(unsigned tie, int a, int n, int m) {
  return ((tie >> (2 * a)) & 1u) && n + 1 >= m ? 1u << (2 * a) : 0u;
}

// A candidate flagged near faces (tie, two bits per axis) may lie, in the FP64 walk, in a cell
// across the flagged faces. True when every such cell rejects it by more than the ratio's
// rounding: the FP64 walk then goes on identically, and only the cell of this candidate's W
// may differ. False when an alternative lies beyond a wall (hit) or any cell may accept.
// st_a: the cell index step of one more face along axis a (s_a times the axis stride).
__device__ __forceinline__ bool all_reject(const float* ratio, int ncells, int cell, unsigned tie, unsigned hit, int st0,
                                           int st1, int st2, float u) {
  if (tie & hit) return false;
#pragma unroll 1
  for (unsigned k = 0; k < 8u; ++k) {
    int c = cell;
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (!((k >> a) & 1u)) continue;
      const unsigned t = (tie >> (2 * a)) & 3u;
      const int st = a == 0 ? st0 : (a == 1 ? st1 : st2);
      ok = ok && t != 0u;
      c += t == 1u ? st : -st;
    }
    if (!ok) continue;
    if (c < 0 || c >= ncells || !(u - ratio[c] >= TIE_ACC)) return false;
  }
  return true;
}

enum { CAND_NULL = 0, CAND_REAL = 1, CAND_DEFER = 2 };

// Adds n units of q to the fixed-point sum of a face.
__device__ __forceinline__ void add_units(long long* Fi, long long face, long long n) {
  atomicAdd(reinterpret_cast<unsigned long long*>(&Fi[face]), (unsigned long long)n);
}

// Outcome of the candidate at path length f.D, whose face counts fb and cell the caller took
// in FP32 (the first wall lies beyond it by more than the bound, so it is a candidate for the
// FP64 walk too): CAND_NULL or CAND_REAL when the FP64 walk decides the same, CAND_DEFER
// otherwise. A candidate whose acceptance draw exceeds the largest ratio of its cell's
// neighbourhood (by more than the ratio's rounding) is rejected wherever it lies, and needs no
// face test; its W may sit in the neighbouring cell. ub: the acceptance word; sy, sz: cell
// index steps along y and z.
// all_real: every candidate of the band is real, and near tells whether a count lies within
// the bound of a face (count_near); otherwise the tie bits are found here when needed.
template <int DIM>
__device__ __forceinline__ int candidate_outcome(const SweepArgs& A, long long bcbase, int ncells, const PW& f,
                                                 float base, int fb0, int fb1, int fb2, int cell, bool all_real,
                                                 bool near, uint32_t ub, int n0, int n1, int n2, int sy, int sz) {
  if (all_real) return near ? CAND_DEFER : CAND_REAL;
  const float ua = word_uniform<float>(ub);
  if (ua - A.ratio_nb32[bcbase + cell] >= TIE_ACC) return CAND_NULL;
  unsigned tie = tie_bits(f.D, f.t0, f.d0, base, fb0, 0);
  if (DIM >= 2) tie |= tie_bits(f.D, f.t1, f.d1, base, fb1, 2);
  if (DIM == 3) tie |= tie_bits(f.D, f.t2, f.d2, base, fb2, 4);
  const float ra = A.ratio32[bcbase + cell];
  if (tie) {
    unsigned hit = tie_hits_wall(tie, 0, fb0, faces_to_wall(f.i0, f.s0, n0));
    if (DIM >= 2) hit |= tie_hits_wall(tie, 1, fb1, faces_to_wall(f.i1, f.s1, n1));
    if (DIM == 3) hit |= tie_hits_wall(tie, 2, fb2, faces_to_wall(f.i2, f.s2, n2));
    if (!all_reject(A.ratio32 + bcbase, ncells, cell, tie, hit, f.s0, f.s1 * sy, f.s2 * sz, ua)) return CAND_DEFER;
  }
  if (fabsf(ua - ra) < TIE_ACC) return CAND_DEFER;
  return ua < ra ? CAND_REAL : CAND_NULL;
}

}  // namespace iugkp
