// Where the FP32 positions of landing.cuh hold, in plain C++ (host and device): the rule by which a
// context's sizes are taken for them, and the test that leaves a candidate to the FP64 walk.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define IUGKP_HD __host__ __device__ __forceinline__
#else
#define IUGKP_HD inline
#endif

namespace iugkp {

// True unless a position lies farther than tol from both faces of its cell (fr: its fraction of the
// cell, one_minus: 1 - fr). Written as the negation of "farther", so that a position or a bound that
// has left FP32 (infinite or NaN) is near: its cell is not used.
IUGKP_HD bool face_near(float fr, float one_minus, float tol) { return !(fminf(fr, one_minus) > tol); }

// A length (cell size, v tau_maj) that the positions may be formed with. Quotients of two of them
// lie within 2^120 of one, a path of 2^20 candidates below 2^85, and a bound |g| (D 2^-19) below
// 2^126: all inside FP32, and cell sizes and their reciprocals are normal numbers with 24 bits. (A
// position X = g D itself may overflow: then it is beyond a wall by more than its bound, as it is.)
IUGKP_HD bool fp32_length(double x) { return x >= 0x1p-60 && x <= 0x1p60; }

}  // namespace iugkp
