// Where candidates lie: emission and landing cells in FP32 with a bound on their distance from
// the FP64 walk's positions, shared by the landing sweeps (land.cu) and the filtered FP64 sweep
// (exact.cu).
//
// A particle's path from emission to its end is one straight segment, so a candidate at path
// length D lies, along axis a, X_a = xi_a + g_a D cells from the emission cell's low face
// (g_a = s_a / h_a): its cell is floor(X_a), and it lies outside the domain exactly when the
// segment met a wall before it.
//
// FP32 against FP64: g_a is within 3.5 2^-23 of its FP64 value (square root 0.75, sincospif
// 0.73, their product 0.5, 1 / h and its product 1.5, in units of 2^-23; walk_bounds_kernel
// measures the first two), D within eD (walk32.cuh), and the sum is rounded once, so X_a is
// within |g_a| D 2^-21 + |g_a| eD + 2^-24 of the FP64 walk's position. LAND_REL and LAND_ABS
// take twice and four times that. A candidate within the bound of a face or a wall is left to
// the FP64 replay, so every real collision is the FP64 walk's. The walls are tested by the
// differences X - lo and X - hi, which are exact where X is near the wall (adding tol to the
// wall's coordinate would round by more than tol on a wide grid).
#pragma once

#include <cuda_runtime.h>

#include "device.cuh"
#include "fp32_range.h"
#include "staged.h"
#include "walk32.cuh"

namespace iugkp {

constexpr float LAND_REL = 0x1p-20f;
constexpr float LAND_ABS = 0x1p-22f;
constexpr float FLOOR_MAGIC = 12582912.f;  // 1.5 2^23: a round-down add leaves floor(X) in the low bits, |X| < 2^22

// Position of a candidate along one axis: its cell offset and whether it lies within tol of a
// face (either side). Where v tau_maj overflows FP32, X and tol are infinite and the offset is
// no cell's: near then (face_near).
__device__ __forceinline__ int floor_near(float X, float tol, bool& near) {
  const float Y = __fadd_rd(X, FLOOR_MAGIC);
  const float fr = X - (Y - FLOOR_MAGIC);
  near |= face_near(fr, 1.f - fr, tol);
  return __float_as_int(Y) - 0x4B400000;
}

// Cell of an emitter of kind `kind` (0: cells; 1 + w: faces of wall w), and for a wall the
// index of its face within the instance.
template <int DIM>
__device__ __forceinline__ void emitter_cell(const InstDesc& in, const StagedArgs& S, int k, int kind, int e, int (&c)[3],
                                             uint32_t& id) {
  const int n0 = in.n[0], n1 = in.n[1], n2 = in.n[2];
  c[0] = c[1] = c[2] = 0;
  if (kind == 0) {
    id = (uint32_t)e;
    if (DIM == 1) {
      c[0] = e;
      return;
    }
    const int r = (int)udiv((unsigned)e, (unsigned)n0, S.mag_n0[k]);
    c[0] = e - r * n0;
    c[1] = r;
    if (DIM == 3) {
      c[2] = (int)udiv((unsigned)r, (unsigned)n1, S.mag_n1[k]);
      c[1] = r - c[2] * n1;
    }
    return;
  }
  const int wl = kind - 1, a = wl >> 1, side = wl & 1;
  // faces of wall a run over (o1, o2) = ((a+1)%3, (a+2)%3), o1 fastest
  const int no1 = a == 0 ? n1 : (a == 1 ? n2 : n0);
  const int j2 = (int)udiv((unsigned)e, (unsigned)no1, S.mag_wall[k * 3 + a]);
  const int j1 = e - j2 * no1;
  long long face;
  if (a == 0) {
    c[0] = side ? n0 - 1 : 0;
    c[1] = j1;
    c[2] = j2;
    face = in.fax_off[0] + (side ? n0 : 0) + (long long)(n0 + 1) * (j1 + (long long)n1 * j2);
  } else if (a == 1) {
    c[0] = j2;
    c[1] = side ? n1 - 1 : 0;
    c[2] = j1;
    face = in.fax_off[1] + j2 + (long long)n0 * ((side ? n1 : 0) + (long long)(n1 + 1) * j1);
  } else {
    c[0] = j1;
    c[1] = j2;
    c[2] = side ? n2 - 1 : 0;
    face = in.fax_off[2] + j1 + (long long)n0 * (j2 + (long long)n1 * (side ? n2 : 0));
  }
  id = (uint32_t)(in.ncells + face);
}

// Direction and fractions within the emission cell from the stream's first block(s); st.j is
// set to the first uniform after the emission.
template <int DIM>
__device__ __forceinline__ void emit_segment(Stream& st, int kind, float (&xi)[3], float (&s)[3]) {
  xi[0] = xi[1] = xi[2] = 0.5f;
  s[0] = s[1] = s[2] = 0.f;
  if (kind == 0) {
    float u_mu, u_phi = 0.5f;
    xi[0] = word_uniform<float>(st.buf.x);
    if (DIM == 1) {
      u_mu = word_uniform<float>(st.buf.y);
    } else if (DIM == 2) {
      xi[1] = word_uniform<float>(st.buf.y);
      u_mu = word_uniform<float>(st.buf.z);
      u_phi = word_uniform<float>(st.buf.w);
    } else {
      xi[1] = word_uniform<float>(st.buf.y);
      xi[2] = word_uniform<float>(st.buf.z);
      u_mu = word_uniform<float>(st.buf.w);
      st.load_block(1);
      u_phi = word_uniform<float>(st.buf.x);
    }
    const float mu = 2.f * u_mu - 1.f;
    s[0] = mu;
    if (DIM >= 2) {
      const float sn = sqrtf(fmaf(-mu, mu, 1.f));
      float sp, cp;
      sincospif(2.f * u_phi, &sp, &cp);
      s[1] = sn * cp;
      s[2] = sn * sp;
    }
    st.j = thermal_uniforms(DIM);
    return;
  }
  const int wl = kind - 1, a = wl >> 1, side = wl & 1;
  float u_n, u_phi = 0.5f, t0 = 0.5f, t1 = 0.5f;
  if (DIM == 1) {
    u_n = word_uniform<float>(st.buf.x);
  } else {
    t0 = word_uniform<float>(st.buf.x);
    if (DIM == 2) {
      u_n = word_uniform<float>(st.buf.y);
      u_phi = word_uniform<float>(st.buf.z);
    } else {
      t1 = word_uniform<float>(st.buf.y);
      u_n = word_uniform<float>(st.buf.z);
      u_phi = word_uniform<float>(st.buf.w);
    }
  }
  const float mn = sqrtf(u_n), sn = DIM >= 2 ? sqrtf(1.f - u_n) : 0.f;
  float sp = 0.f, cp = 0.f;
  if (DIM >= 2) sincospif(2.f * u_phi, &sp, &cp);
  const float nrm = side ? -mn : mn, ta = sn * cp, tb = sn * sp, edge = side ? 1.f : 0.f;
  if (a == 0) {
    s[0] = nrm; s[1] = ta; s[2] = tb;
    xi[0] = edge; xi[1] = t0; xi[2] = t1;
  } else if (a == 1) {
    s[1] = nrm; s[2] = ta; s[0] = tb;
    xi[1] = edge; xi[0] = t0; xi[2] = t1;
  } else {
    s[2] = nrm; s[0] = ta; s[1] = tb;
    xi[2] = edge; xi[0] = t0; xi[1] = t1;
  }
  st.j = wall_uniforms(DIM);
}

// One lane's emitter of a landing task: its rank in the group's visiting order, emitter index,
// cell, stream identity and weight (per unit emission temperature when ADJ), and the distances
// to the walls in cells. `on` is false for lanes without an emitter and for zero weights.
template <int DIM>
struct LaneEmitter {
  int rank, e, sub, cell0;
  uint32_t id;
  double w;
  bool has, on;
  float ih[3], lo[3], hi[3];
  int c[3];
  // The emitter's weight in the group's band.
  template <bool ADJ>
  __device__ __forceinline__ void weight(const SweepArgs& A, const LandGroup& G, const InstDesc& in) {
    if (G.kind == 0) {
      w = A.coef[in.bc_off + (long long)G.band * in.ncells + e];
      if (!ADJ) {
        double Te = A.T[in.cell_off + e];
        if (A.srcshift) Te += A.srcshift[in.cell_off + e];
        w *= Te;
      }
    } else {
      w = A.wcoef[(long long)(G.inst * A.nb + G.band) * 6 + G.kind - 1];
      if (!ADJ) w *= A.wallTf[in.bface_off + in.wface_off[G.kind - 1] + e];
    }
    on = has && (__double_as_longlong(w) << 1) != 0;  // +-0: nothing to trace
  }
  template <bool ADJ>
  __device__ __forceinline__ void init(const SweepArgs& A, const StagedArgs& S, const LandGroup& G, const InstDesc& in,
                                       int tile, int lane) {
    sub = lane / G.tw;
    rank = tile * G.tw + lane - sub * G.tw;
    has = sub < G.reps && rank < G.ne;
    e = has ? rank : 0;
    if (G.perm_off >= 0) e = A.perm[G.perm_off + e];
    emitter_cell<DIM>(in, S, G.inst, G.kind, e, c, id);
    weight<ADJ>(A, G, in);
    const int n0 = in.n[0], n1 = in.n[1], n2 = in.n[2];
#pragma unroll
    for (int a = 0; a < DIM; ++a) {
      ih[a] = __frcp_rn(in.hf[a]);
      lo[a] = (float)-c[a];
      hi[a] = (float)((a == 0 ? n0 : (a == 1 ? n1 : n2)) - c[a]);
    }
    cell0 = c[0] + n0 * (c[1] + n1 * c[2]);
  }
};

// The group of a claimed task, kept until a task of another group comes.
struct TaskGroup {
  unsigned t_beg = 1, t_end = 0;  // tasks of the cached group
  int gi = 0;
  __device__ __forceinline__ void find(const LandArgs& L, unsigned task) {
    if (task >= t_beg && task < t_end) return;
    int lo = 0, hi = L.n_groups - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (L.groups[mid].task0 <= task) lo = mid;
      else hi = mid - 1;
    }
    gi = lo;
    t_beg = L.groups[lo].task0;
    t_end = lo + 1 < L.n_groups ? L.groups[lo + 1].task0 : L.n_tasks;
  }
};

}  // namespace iugkp
