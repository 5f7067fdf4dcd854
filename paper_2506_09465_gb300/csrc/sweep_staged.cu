// Fast forward sweep in 1D and 2D (3D: sweep_chain.cu): FP32 walk, persistent blocks (a
// pass-synchronous kernel for 2D, a per-lane-refill kernel for both), face tallies staged in
// shared memory in fixed point. Same method and draws as the plain sweep
// (arXiv 2506.09465 Sec. 3.1 steps (1)-(3), Sec. 3.2 null collisions); only the
// arithmetic precision of the walk and the way tallies are accumulated differ.
//
// Face tallies:
//  * faces normal to x are accumulated in a shared-memory copy of the instance's x-faces
//    (all of them when they fit, else a centred run), as integers in units of
//    q = w_max 2^-26 (exact and independent of the order of the additions): 32-bit words
//    (native shared-memory atomics, about five times the rate of 64-bit ones) whose rare
//    wrap-arounds add +-2^32 q to the FP64 face at once, flushed to the FP64 array when the
//    block leaves the instance; x-faces outside the window take global atomics;
//  * faces normal to y in 2D are not tallied, except on the low
//    boundary: every particle conserves power, so in every cell the net inflow equals the
//    absorbed minus emitted power, and the last-axis faces follow exactly by a prefix sum
//    along each column (close_2d_kernel);
//  * 2D instances whose faces all fit the window use two-group tallies instead: a particle
//    tallies only the faces normal to the axis it crosses less often, and each group's
//    other faces follow from that group's own per-cell balance (close_2d_kernel);
//  * a warp tallies the face items of the particles that ended together: in the
//    pass-synchronous kernel each lane takes segments of 8 items of one list, dealt
//    round-robin; in the 2D per-lane-refill kernel each lane takes one contiguous chunk of the
//    concatenated item lists;
//  * nothing is tallied per particle for the walls: the power a wall emits enters through
//    its faces deterministically (N particles of known weight per face), and the power it
//    absorbs follows from its faces (closing.cu).
#include <cuda_runtime.h>

#include <algorithm>

#include "device.cuh"
#include "internal.h"
#include "landing.cuh"
#include "segment.cuh"
#include "staged.h"
#include "walk32.cuh"

namespace iugkp {

// Per-lane cache of the group of the lane's previous particle (and of the weight of a
// wall group, which is the same for all its particles).
struct EmitCache {
  unsigned g_first, g_end;  // forward particle range of the cached group
  int g_ne, g_kind, g_band;
  int g_perm;               // perm_off of the group
  unsigned g_mag;           // division magic of n_emitters
  int e;
  double w;
};

// Emits forward particle pid into the lane state. Returns false for a zero-weight
// particle (nothing to trace).
template <int DIM>
__device__ __forceinline__ bool staged_emit(const SweepArgs& A, const StagedArgs& S, unsigned pid, double& w,
                                            int& band, PW& f, Stream& st, uint32_t& ub, EmitCache& ec,
                                            const InstDesc& in, int k, bool two) {
  if (pid < ec.g_first || pid >= ec.g_end) {
    const int gi = find_group(A.groups, A.n_groups, (long long)pid);
    const Group G = A.groups[gi];
    ec.g_first = (unsigned)G.first_particle;
    ec.g_end = (unsigned)(G.first_particle + (long long)G.n_emitters * G.per_emitter);
    ec.g_ne = G.n_emitters;
    ec.g_kind = G.kind;
    ec.g_band = G.band;
    ec.g_mag = S.group_mag[gi];
    ec.g_perm = G.perm_off;
    ec.e = -1;
  }
  band = ec.g_band;
  const int b = ec.g_band;
  // The staged sweep visits a group's particles q-major (particle q of every emitter,
  // then q + 1), so the lanes of a warp start in different cells: their face and deposit
  // tallies rarely hit the same address at the same time; within a q the emitters come in
  // the group's visiting order. Draws are keyed by (emitter, particle), so the order changes
  // nothing else.
  const unsigned local = pid - ec.g_first;
  const int q = (int)udiv(local, (unsigned)ec.g_ne, ec.g_mag);
  int e = (int)(local - (unsigned)q * (unsigned)ec.g_ne);
  if (ec.g_perm >= 0) e = A.perm[ec.g_perm + e];
  const int n0 = in.n[0], n1 = in.n[1];
  const int kind = ec.g_kind;
  float xi0 = 0.5f, xi1 = 0.5f, sx = 0.f, sy = 0.f;
  if (kind == 0) {
    w = A.wemit[in.bc_off + (long long)b * in.ncells + e];  // from the pass before the trace
    if ((__double_as_longlong(w) << 1) == 0) return false;   // +-0: nothing to trace
    st.init(A.seed, in.inst_id, (uint32_t)b, A.epoch, (uint32_t)e, (uint32_t)q);
    if (DIM == 1) {
      f.i0 = e;
      f.i1 = 0;
    } else {
      const int r = (int)udiv((unsigned)e, (unsigned)n0, S.mag_n0[k]);
      f.i0 = e - r * n0;
      f.i1 = r;
    }
    float u_mu, u_phi = 0.5f;
    if (DIM == 1) {
      xi0 = word_uniform<float>(st.buf.x);
      u_mu = word_uniform<float>(st.buf.y);
    } else {
      xi0 = word_uniform<float>(st.buf.x);
      xi1 = word_uniform<float>(st.buf.y);
      u_mu = word_uniform<float>(st.buf.z);
      u_phi = word_uniform<float>(st.buf.w);
    }
    const float mu = 2.f * u_mu - 1.f;
    sx = mu;
    if (DIM >= 2) {
      const float sn = sqrtf(fmaf(-mu, mu, 1.f));  // 1 - mu^2 with one rounding
      float sp, cp;
      sincospif(2.f * u_phi, &sp, &cp);
      sy = sn * cp;
    }
    st.j = thermal_uniforms(DIM);
  } else {
    const int wl = kind - 1;
    if (ec.e != -2) {
      ec.w = A.wcoef[((long long)k * A.nb + b) * 6 + wl];  // per unit face temperature
      ec.e = -2;
    }
    w = ec.w * A.wallTf[in.bface_off + in.wface_off[wl] + e];
    if (w == 0.0) return false;
    const int a = wl >> 1, side = wl & 1;
    long long face;  // a wall's faces run along the other axis (1D: one face)
    if (a == 0) {
      f.i0 = side ? n0 - 1 : 0;
      f.i1 = e;
      face = in.fax_off[0] + (side ? n0 : 0) + (long long)(n0 + 1) * e;
    } else {
      f.i0 = e;
      f.i1 = side ? n1 - 1 : 0;
      face = in.fax_off[1] + e + (long long)n0 * (side ? n1 : 0);
    }
    st.init(A.seed, in.inst_id, (uint32_t)b, A.epoch, (uint32_t)(in.ncells + face), (uint32_t)q);
    float u_n, u_phi = 0.5f;
    float t0 = 0.5f;  // tangential fraction
    if (DIM == 1) {
      u_n = word_uniform<float>(st.buf.x);
    } else {
      t0 = word_uniform<float>(st.buf.x);
      u_n = word_uniform<float>(st.buf.y);
      u_phi = word_uniform<float>(st.buf.z);
    }
    const float mn = sqrtf(u_n);
    const float sn = DIM >= 2 ? sqrtf(1.f - u_n) : 0.f;
    float sp = 0.f, cp = 0.f;
    if (DIM >= 2) sincospif(2.f * u_phi, &sp, &cp);
    // the wall's tangential axes are (a+1)%3 (cosine) and (a+2)%3 (sine)
    if (a == 0) {
      sx = side ? -mn : mn;
      sy = sn * cp;
      xi0 = side ? 1.f : 0.f;
      xi1 = t0;
    } else {
      sy = side ? -mn : mn;
      sx = sn * sp;
      xi1 = side ? 1.f : 0.f;
      xi0 = t0;
    }
    st.j = wall_uniforms(DIM);  // (the power entering through wall faces is added after the trace)
  }
  axis_init(sx, xi0, in.hf[0], f.t0, f.d0, f.s0);
  f.tex = axis_exit(f.i0, f.s0, n0, f.t0, f.d0);
  if (DIM >= 2) {
    axis_init(sy, xi1, in.hf[1], f.t1, f.d1, f.s1);
    const float e1 = axis_exit(f.i1, f.s1, n1, f.t1, f.d1);
    // the axis of the wall the segment reaches (x on ties), kept in the unused i2
    f.i2 = e1 < f.tex ? 1 : 0;
    f.tex = fminf(f.tex, e1);
  }
  if (DIM == 2 && two && f.d0 < f.d1) {
    // y-group: its emission enters its own power balance (cell) or boundary flux (face)
    if (kind == 0) {
      atomicAdd(&S.DY[in.cell_off + e], -w);
    } else {
      const int wl = kind - 1;
      atomicAdd(&S.EY[in.bface_off + in.wface_off[wl] + e], (wl & 1) ? -w : w);
    }
  }
  // the first candidate: its path word from block 0's unused bits; its acceptance word only
  // where some cell of the band may reject (else every candidate is real and the particle ends
  // at its first candidate, so no later draw is taken)
  ub = A.all_real[(long long)k * A.nb + b] ? 0u : st.even_word();
  st.j += 2;
  f.D = __fmul_rn(-__logf(word_uniform<float>(st.first)), A.vtm32[(long long)k * A.nb + b]);
  return true;
}

// Persistent blocks. Each block works on one instance at a time (first the instance its
// index falls on by estimated cost, then any instance with work left); its warps take
// private ranges of the instance's particles and refill idle lanes together. Faces normal
// to x go to a shared-memory copy of the instance's x-faces (when it fits), in units of
// the instance's q; the block flushes it when it leaves the instance.
// FP64 value of compensated tallies: dst = hi + lo (add = 0) or dst += hi + lo (add = 1).
__global__ void k32_finalize_kernel(const float2* src, double* dst, long long n, int add) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float2 v = src[i];
    const double x = (double)v.x + (double)v.y;
    dst[i] = add ? dst[i] + x : x;
  }
}

template <int DIM, bool K32>
__global__ void __launch_bounds__(STAGED_NT, 1) sweep_staged_kernel(SweepArgs A, StagedArgs S) {
  extern __shared__ unsigned win[];
  // cooperative tallies: per warp, each lane's particle parameters and the item list starts
  __shared__ int4 s_par[STAGED_NT / 32][64];
  __shared__ int s_lst[STAGED_NT / 32][33];
  __shared__ int s_inst;
  LCounts cnt;
#pragma unroll
  for (int k = 0; k < CNT_N; ++k) cnt.v[k] = 0;
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  const bool useF = A.F != nullptr;
  const int n_inst = S.n_inst;
  int start = 0;
  {
    const double pos = (blockIdx.x + 0.5) / gridDim.x * S.cost_total;
    while (start + 1 < n_inst && S.cost_prefix[start + 1] <= pos) ++start;
  }
  for (int visit = 0; visit < n_inst; ++visit) {
    const int k = (start + visit) % n_inst;
    if (threadIdx.x == 0) s_inst = (*(volatile unsigned long long*)&S.inst_next[k] < (unsigned long long)S.inst_end[k]) ? k : -1;
    __syncthreads();
    if (s_inst < 0) {
      __syncthreads();
      continue;
    }
    const InstDesc& in = A.inst[k];
    // descriptor fields used inside the walk, held in registers (the atomics below would
    // otherwise force reloads)
    const int n0 = in.n[0], n1 = in.n[1];
    const long long face_off = in.face_off, fax1 = in.fax_off[1];
    const long long bc_off = in.bc_off;
    const int ncells = in.ncells, refill = S.refill > 0 ? S.refill : in.refill;
    const int sy_cell = n0, sy_xf = n0 + 1;  // cell and x-face index steps along y
    // x-faces [wbase, wbase + wlen) of this instance are tallied in the shared window
    const int2 wd = useF ? S.window[k] : make_int2(0, 0);
    const int wbase = wd.x;
    const unsigned wlen = (unsigned)wd.y;
    const bool wfull = wbase == 0 && (long long)wlen == (long long)(n0 + 1) * n1;
    // 2D instance whose faces all fit the window: two-group tallies (see StagedArgs)
    const bool two = DIM == 2 && useF && wbase == 0 && (long long)wlen == in.nfaces;
    for (unsigned i = threadIdx.x; i < wlen; i += STAGED_NT) win[i] = WIN_BIAS;
    __syncthreads();
    const double qinv = S.wmax[k] > 0.0 ? WIN_SCALE / S.wmax[k] : 0.0;
    const unsigned pend = (unsigned)S.inst_end[k];
    unsigned rbeg = 0, rend = 0;  // this warp's private particle range
    double w = 0.0;
    unsigned qwx = 0;             // signed x-face contribution in units of q (two's complement)
    int band = 0;
    long long bcbase = 0;
    float vtm = 0.f;
    PW f;
    Stream st;
    uint32_t ub = 0;
    bool alive = false, exhausted = false;
    bool tally = false;     // the lane's particle has ended and tallies its faces
    int kcur = 0, kend = 0; // face items of the tally phase
    EmitCache ec;
    ec.g_first = 1;
    ec.g_end = 0;  // empty: forces a lookup on the first emission
    ec.e = -1;
    float eD = 0.f;         // bound of |D - D_fp64| of the lane's particle
    int kc = 0;             // its candidates tallied so far
    unsigned pid = 0;       // its forward index
    for (;;) {
      // ---- refill idle lanes together ----
      const unsigned dead = __ballot_sync(0xffffffffu, !alive);
      if (!exhausted && __popc(dead) >= refill) {
        if (rbeg == rend) {  // private range used up: take the next one of the instance
          unsigned long long got = 0;
          if (lane == 0) got = atomicAdd(&S.inst_next[k], (unsigned long long)S.warp_grab);
          got = __shfl_sync(0xffffffffu, got, 0);
          if (got < pend) {
            rbeg = (unsigned)got;
            rend = (unsigned)min(got + (unsigned long long)S.warp_grab, (unsigned long long)pend);
          } else {
            exhausted = true;
          }
        }
        const unsigned rank = __popc(dead & lt_mask);
        const unsigned take = min((unsigned)__popc(dead), rend - rbeg);
        if (!alive && rank < take) {
          alive = staged_emit<DIM>(A, S, rbeg + rank, w, band, f, st, ub, ec, in, k, two);
          if (alive) {
            cnt.v[CNT_FLIGHTS] += 1;
            // round(w / q) as the low word of w qinv + 1.5 2^52 (one FMA, |w qinv| <= 2^26)
            const int qw = __double2loint(fma(w, qinv, 0x1.8p52));
            // signed along the axis whose faces the particle tallies
            qwx = (unsigned)(((two && f.d0 < f.d1) ? f.s1 : f.s0) > 0 ? qw : -qw);
            vtm = A.vtm32[(long long)k * A.nb + band];
            bcbase = bc_off + (long long)band * ncells;
            eD = fmaf(f.D, TIE_LOG_REL, vtm * TIE_LOG_ABS);
            kc = 0;
            pid = rbeg + rank;
          }
        }
        rbeg += take;
      }
      if (!__any_sync(0xffffffffu, alive)) {
        if (exhausted) break;
        continue;
      }
      // ---- candidates (Sec. 3.2): up to walk_k per lane. The candidate lies at path length D
      // of the straight segment; its cell follows from the faces before D on each axis.
      // W tally, then acceptance with probability tau_maj / tau(x); a rejected candidate
      // draws the next flight length and the particle goes on in the same direction ----
      int nitem = 0;  // cooperative tallies: face items of the lane's particle ended in this pass
      bool ended = false, wall_exit = false, deferred = false;
      const bool walking = alive && !tally;
      const bool all_real = A.all_real[(long long)k * A.nb + band] != 0;
      if (walking) {
#pragma unroll 1
        for (int it = 0; it < S.walk_k; ++it) {
          // a decision within rounding of the FP64 walk's defers the particle to the FP64 replay
          const float base = fmaf(TIE_REL, f.D, eD);
          if (f.D - f.tex > base) {  // the segment reaches a wall first: absorbed there
            ended = wall_exit = true;
            break;
          }
          if (f.tex - f.D <= fmaf(TIE_REL, f.tex, eD)) {  // at the first wall within rounding
            ended = deferred = true;
            break;
          }
          bool near = false;  // a count within the bound of a face, found with it for all-real bands
          int fb0, fb1 = 0;
          if (all_real) {
            fb0 = count_near(f.D, f.t0, f.d0, base, near);
            if (DIM >= 2) fb1 = count_near(f.D, f.t1, f.d1, base, near);
          } else {
            fb0 = faces_before(f.D, f.t0, f.d0);
            if (DIM >= 2) fb1 = faces_before(f.D, f.t1, f.d1);
          }
          int cell = clampi(f.i0 + f.s0 * fb0, n0);
          if (DIM >= 2) cell += sy_cell * clampi(f.i1 + f.s1 * fb1, n1);
          const long long ci = bcbase + cell;
          const int oc = candidate_outcome<DIM>(A, bcbase, ncells, f, base, fb0, fb1, 0, cell, all_real, near, ub,
                                                n0, n1, 1, sy_cell, 0);
          if (oc == CAND_DEFER) {
            ended = deferred = true;
            break;
          }
          cnt.v[CNT_CANDIDATES] += 1;
          ++kc;
          // W collects w here; the sweep scales it by tau_maj afterwards, and
          // a band whose every candidate is real takes W = tau_maj R there instead
          if (K32 && S.W32 && !all_real) tally_k32(&S.W32[ci], w);
          else if (!K32 && A.W && !all_real) atomicAdd(&A.W[ci], w);
          if (oc == CAND_REAL) {
            cnt.v[CNT_REAL] += 1;
            if (K32) {
              tally_k32(&S.R32[ci], w);
            } else {
              atomicAdd(&A.R[ci], w);
            }
            if (two && f.d0 < f.d1) atomicAdd(&S.DY[in.cell_off + cell], w);
            ended = true;
            break;
          }
          uint32_t uw;
          st.next_pair(uw, ub);
          const float ell = __fmul_rn(-__logf(word_uniform<float>(uw)), vtm);
          f.D = __fadd_rn(f.D, ell);
          eD = fmaf(f.D, TIE_SUM, fmaf(ell, TIE_LOG_REL, eD + vtm * TIE_LOG_ABS));
        }
      }
      if (walking) {
        if (deferred) {
          defer_particle(S, pid, ((unsigned)kc << 1) | ((two && f.d0 < f.d1) ? 1u : 0u));
          ended = false;
          alive = false;
        }
        if (ended) {
          // interior faces crossed before the end, per axis; on the exit axis the wall face
          // lies exactly at tex, so its count is known without rounding
          const float L = wall_exit ? f.tex : f.D;
          int ex = -1;
          if (wall_exit) {
            const float e0 = axis_exit(f.i0, f.s0, n0, f.t0, f.d0);
            const float e1 = DIM >= 2 ? axis_exit(f.i1, f.s1, n1, f.t1, f.d1) : INFINITY;
            ex = e0 <= e1 ? 0 : 1;
          }
          // at a wall, the faces of the other axes crossed before it: a count within rounding
          // of the FP64 walk's (the segment leaves near a cell corner) defers the particle
          bool tie = false;
          const float bx = TIE_REL * f.tex;
          const int m0 = faces_to_wall(f.i0, f.s0, n0);
          int c0 = m0 - 1, c1 = 0, m1 = 1;
          if (ex != 0) {
            const int q = count_near(L, f.t0, f.d0, bx, tie);
            c0 = min(q, m0 - 1);
          }
          if (DIM >= 2) {
            m1 = faces_to_wall(f.i1, f.s1, n1);
            c1 = m1 - 1;
            if (ex != 1) {
              const int q = count_near(L, f.t1, f.d1, bx, tie);
              c1 = min(q, m1 - 1);
            }
          }
          if (wall_exit && tie) {
            defer_particle(S, pid, ((unsigned)kc << 1) | ((two && f.d0 < f.d1) ? 1u : 0u));
            alive = false;
          } else {
            if (wall_exit) cnt.v[CNT_WALL_EXITS] += 1;
            cnt.v[CNT_CROSSINGS] += c0 + c1;
            if (DIM == 2 && (two || wfull)) {
              // Face items k = 0 .. kend-1 along the tallied axis p (the other axis: q). Item k
              // is the face index a0 + k sp + sq min(ceil(u0 + k r), lim): the k-th face normal
              // to p, in the row (or column) given by the faces normal to q crossed before it,
              // ceil(u0 + k r) with u0 = (t_p - t_q) / d_q and r = d_p / d_q, at most lim.
              const bool yg = two && f.d0 < f.d1;
              int a0, sp, sq, lim;
              float u0, r;
              if (!yg) {
                // exit through the low y-wall: the one face normal to y this group tallies
                if (ex == 1 && f.s1 < 0) {
                  const int col = f.i0 + f.s0 * c0;
                  atomicAdd(&S.gx()[in.bface_off + in.wface_off[2] + col], -w);
                }
                kend = c0 + (ex == 0 ? 1 : 0);
                const bool flat = !(f.d1 < INFINITY);
                u0 = flat ? -1.f : __fdividef(f.t0 - f.t1, f.d1);
                r = flat ? 0.f : __fdividef(f.d0, f.d1);
                lim = m1 - 1;
                a0 = (f.s0 > 0 ? f.i0 + 1 : f.i0) + sy_xf * f.i1;
                sp = f.s0;
                sq = f.s1 * sy_xf;
              } else {
                // exit through the low x-wall: the one face normal to x this group tallies
                if (ex == 0 && f.s0 < 0) atomicAdd(&S.gx()[in.bface_off + in.wface_off[0] + (f.i1 + f.s1 * c1)], -w);
                kend = c1 + (ex == 1 ? 1 : 0);
                u0 = __fdividef(f.t1 - f.t0, f.d0);
                r = __fdividef(f.d1, f.d0);
                lim = m0 - 1;
                a0 = (int)fax1 + f.i0 + n0 * (f.s1 > 0 ? f.i1 + 1 : f.i1);
                sp = f.s1 * n0;
                sq = f.s0;
              }
              f.i0 = a0;
              f.s0 = sp;
              f.s1 = sq;
              f.i2 = lim;
              f.D = u0;
              f.tex = r;
              nitem = kend;  // tallied below by the whole warp
              alive = false;
            } else if (useF) {
              // faces normal to the last axis: only the low boundary is tallied (the rest
              // follow from conservation)
              if (DIM == 2 && ex == 1 && f.s1 < 0) {
                atomicAdd(&S.gx()[in.bface_off + in.wface_off[2] + (f.i0 + f.s0 * c0)], -w);
              }
              // x-faces crossed (the wall face too when the particle leaves through x)
              kcur = 0;
              kend = c0 + (ex == 0 ? 1 : 0);
              if (DIM == 2) {
                // rows of the x-face crossings, incrementally: faces normal to y before the
                // k-th x-face = ceil(u0 + k r), u0 = (t0 - t1) / d1, r = d0 / d1
                const bool flat = !(f.d1 < INFINITY);
                f.D = flat ? -1.f : __fdividef(f.t0 - f.t1, f.d1);
                f.tex = flat ? 0.f : __fdividef(f.d0, f.d1);
                f.i2 = m1 - 1;  // largest count of y-faces a row index may take
              }
              tally = kend > 0;
              alive = tally;
            } else {
              alive = false;
            }
          }
        }
      }
      // ---- 2D, every tallied face in the window: the warp tallies the face items of the
      // particles that ended in this pass together. The items are concatenated in lane
      // order and cut into 32 equal contiguous chunks, one per lane; a lane finds the
      // particle holding its first item by binary search over the list starts and reads
      // each particle's parameters from shared memory when its chunk enters that list ----
      if (DIM == 2 && (two || wfull)) {
        int incl = nitem;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += t;
        }
        const int total = __shfl_sync(0xffffffffu, incl, 31);
        if (total > 0) {
          const int first = incl - nitem;
          int4* par = s_par[threadIdx.x >> 5];
          int* lst = s_lst[threadIdx.x >> 5];
          lst[lane] = first;
          if (lane == 31) lst[32] = total;
          if (nitem > 0) {
            par[2 * lane] = make_int4(f.i0, f.s0, f.s1, f.i2);
            par[2 * lane + 1] = make_int4(__float_as_int(f.D), __float_as_int(f.tex), (int)qwx, first);
          }
          __syncwarp();
          const int c0 = (lane * total) >> 5, c1 = ((lane + 1) * total) >> 5;
          if (c0 < c1) {
            // the last list starting at or before c0 (it holds c0: empty lists start where
            // the next one does)
            int l = 0;
#pragma unroll
            for (int st = 16; st > 0; st >>= 1)
              if (lst[l + st] <= c0) l += st;
            int lend = lst[l + 1];
            int4 pa = par[2 * l], pb = par[2 * l + 1];
#pragma unroll 1
            for (int kk = c0; kk < c1; ++kk) {
              if (kk >= lend) {
                do {
                  ++l;
                  lend = lst[l + 1];
                } while (lend <= kk);
                pa = par[2 * l];
                pb = par[2 * l + 1];
              }
              // item kl of the particle: a0 + kl sp + sq min(ceil(u0 + kl r), lim)
              const int kl = kk - pb.w;
              const int face =
                  pa.x + kl * pa.y +
                  pa.z * min(ceil_count(fmaf(small_int_float(kl), __int_as_float(pb.y), __int_as_float(pb.x))), pa.w);
              const unsigned q = (unsigned)pb.z;
              const unsigned old = atomicAdd(&win[face], q);
              // |q| <= 2^26, so the word can wrap only from within 2^26 of 0 / 2^32
              if (old + 0x04000000u < 0x08000000u) {
                const int carry = ((int)q >> 31) + (old + q < old ? 1 : 0);
                if (carry) add_units(S.Fi, face_off + face, (long long)carry << 32);
              }
            }
          }
          __syncwarp();
        }
      }
      // ---- face tallies of ended particles: up to walk_k per lane ----
      if (tally) {
        const int kstop = min(kend, kcur + S.walk_k);
        float fk = small_int_float(kcur);  // the item index in FP32, advanced without conversions
        // 64-bit sums kept as 32-bit low words in the window plus carries added to the FP64
        // face: the old word tells whether an addition wrapped (rare: words start at 2^31
        // and one contribution is at most 2^26)
        auto window_add = [&](int xface, unsigned rel) {
          const unsigned old = atomicAdd(&win[rel], qwx);
          if (old + 0x04000000u < 0x08000000u) {  // a wrap starts within 2^26 of 0 / 2^32
            const int carry = ((int)qwx >> 31) + (old + qwx < old ? 1 : 0);
            if (carry) add_units(S.Fi, face_off + xface, (long long)carry << 32);
          }
        };
        // (2D instances whose tallied faces are all in the window have tallied them above)
#pragma unroll 1
        for (; kcur < kstop; ++kcur, fk += 1.f) {
          int xface = f.s0 > 0 ? f.i0 + 1 + kcur : f.i0 - kcur;
          if (DIM == 2) {
            xface += sy_xf * (f.i1 + f.s1 * min(ceil_count(fmaf(fk, f.tex, f.D)), f.i2));
          }
          const unsigned rel = (unsigned)(xface - wbase);
          if (rel < wlen) window_add(xface, rel);
          else if (K32) tally_k32(&S.F32[face_off + xface], f.s0 > 0 ? w : -w);
          else atomicAdd(&A.F[face_off + xface], f.s0 > 0 ? w : -w);
        }
        if (kcur >= kend) {
          tally = false;
          alive = false;
        }
      }
    }
    __syncthreads();
    for (unsigned i = threadIdx.x; i < wlen; i += STAGED_NT) {  // x-faces come first
      const int v = (int)(win[i] - WIN_BIAS);
      if (v) add_units(S.Fi, face_off + wbase + i, v);
    }
    __syncthreads();
  }
  flush_lcounts(cnt, A.counters);
}

// 2D instances whose tallied faces all sit in the window, pass by pass: every pass of a warp
// emits up to 32 particles (one per lane), follows each to its end (real collision or
// wall), and tallies the face items of all of them together (the cooperative tallies of
// sweep_staged_kernel). A particle's state lives only inside its pass, so the tally loop
// runs with the per-particle registers free. Same particles, draws and tallies as
// sweep_staged_kernel; chosen when the candidates per flight are few (each lane waits for
// the longest flight of its pass). REAL: tau = tau_maj in every cell of every instance and
// band, so every candidate is real and the acceptance test is left out. PARTIAL: some
// instance's x-faces exceed the window (a centred run of them sits there); the faces outside
// take global atomics of the same fixed-point contribution.
template <bool K32, bool REAL, bool PARTIAL>
__global__ void __launch_bounds__(STAGED_NT, 1) sweep_sync_kernel(SweepArgs A, StagedArgs S, SyncArgs Y) {
  extern __shared__ unsigned win[];
  __shared__ int4 s_par[STAGED_NT / 32][64];
  __shared__ int s_lst[STAGED_NT / 32][33];
  __shared__ int s_inst;
  LCounts cnt;
#pragma unroll
  for (int k = 0; k < CNT_N; ++k) cnt.v[k] = 0;
  const int lane = threadIdx.x & 31;
  const int n_inst = S.n_inst;
  int start = 0;
  {
    const double pos = (blockIdx.x + 0.5) / gridDim.x * S.cost_total;
    while (start + 1 < n_inst && S.cost_prefix[start + 1] <= pos) ++start;
  }
  int4* par = s_par[threadIdx.x >> 5];
  int* lst = s_lst[threadIdx.x >> 5];
  TaskGroup tg;
  for (int visit = 0; visit < n_inst; ++visit) {
    const int k = (start + visit) % n_inst;
    const unsigned task_end = Y.task_end[k];
    if (threadIdx.x == 0) s_inst = (*(volatile unsigned long long*)&S.inst_next[k] < (unsigned long long)task_end) ? k : -1;
    __syncthreads();
    if (s_inst < 0) {
      __syncthreads();
      continue;
    }
    const InstDesc& in = A.inst[k];
    const int n0 = in.n[0], n1 = in.n[1];
    const long long face_off = in.face_off, fax1 = in.fax_off[1];
    const int sy_xf = n0 + 1;
    const int wbase = PARTIAL ? S.window[k].x : 0;
    const unsigned wlen = (unsigned)S.window[k].y;
    // every face in the window (two-group tallies); else x-faces [wbase, wbase + wlen)
    const bool two = wbase == 0 && (long long)wlen == in.nfaces;
    for (unsigned i = threadIdx.x; i < wlen; i += STAGED_NT) win[i] = WIN_BIAS;
    __syncthreads();
    const double qinv = S.wmax[k] > 0.0 ? WIN_SCALE / S.wmax[k] : 0.0;
    const float h0 = in.hf[0], h1 = in.hf[1];
    const uint32_t inst_id = in.inst_id;
    const int ncells = in.ncells;
    const long long coff = in.cell_off;
    double* const gx = S.gx() + in.bface_off;
    for (;;) {
      // the next task of the instance: a tile of emitters (one or more lanes each) x a run of
      // particle numbers; the lanes keep their emitters for the run
      unsigned long long got = 0;
      if (lane == 0) got = atomicAdd(&S.inst_next[k], 1ull);
      got = __shfl_sync(0xffffffffu, got, 0);
      if (got >= task_end) break;
      tg.find(Y.L, (unsigned)got);
      const LandGroup& G = Y.L.groups[tg.gi];
      const unsigned tk = (unsigned)got - tg.t_beg;
      const int qc = (int)(tk / (unsigned)G.ntile), tile = (int)(tk - (unsigned)qc * (unsigned)G.ntile);
      const int kind = G.kind, band = G.band;
      const int sub = lane / G.tw, rank = tile * G.tw + lane - sub * G.tw;
      int e = sub < G.reps && rank < G.ne ? rank : 0;
      if (G.perm_off >= 0) e = A.perm[G.perm_off + e];
      int c[3];
      uint32_t id;
      emitter_cell<2>(in, S, k, kind, e, c, id);
      const long long bcbase = in.bc_off + (long long)band * ncells;
      double w;
      if (kind == 0) {
        w = A.wemit[bcbase + e];  // from the pass before the trace
      } else {
        w = A.wcoef[(long long)(k * A.nb + band) * 6 + kind - 1] * A.wallTf[in.bface_off + in.wface_off[kind - 1] + e];
      }
      // +-0: nothing to trace
      const bool on = sub < G.reps && rank < G.ne && (__double_as_longlong(w) << 1) != 0;
      const int qw = __double2loint(fma(w, qinv, 0x1.8p52));
      const float vtm = A.vtm32[k * A.nb + band];
      const bool all_real = REAL || A.all_real[k * A.nb + band] != 0;
      const float ea = vtm * TIE_LOG_ABS;
      const int qbeg = qc * (Y.L.qch * G.reps) + sub, qend = min(G.per, (qc + 1) * (Y.L.qch * G.reps));
      int n_yg = 0;  // the lane's y-group flights of this task: their emission enters its own balance
      for (int pass = 0; pass < Y.L.qch; ++pass) {
        const int q = qbeg + pass * G.reps;
        const bool act = on && q < qend;
        if (!__any_sync(0xffffffffu, act)) break;
        int nitem = 0;
        int4 pa_own, pb_own;  // this lane's item parameters, stored once its list slot is known
        if (act) {
          PW f;
          Stream st;
          uint32_t ub;
          st.init(A.seed, inst_id, (uint32_t)band, A.epoch, id, (uint32_t)q);
          {
            float xi[3], s[3];
            emit_segment<2>(st, kind, xi, s);
            f.i0 = c[0];
            f.i1 = c[1];
            axis_init(s[0], xi[0], h0, f.t0, f.d0, f.s0);
            f.tex = axis_exit(f.i0, f.s0, n0, f.t0, f.d0);
            axis_init(s[1], xi[1], h1, f.t1, f.d1, f.s1);
            const float e1 = axis_exit(f.i1, f.s1, n1, f.t1, f.d1);
            f.i2 = e1 < f.tex ? 1 : 0;  // the axis of the wall the segment reaches (x on ties)
            f.tex = fminf(f.tex, e1);
          }
          const bool yg = two && f.d0 < f.d1;
          n_yg += yg ? 1 : 0;
          // the first candidate: its path word from block 0's unused bits; its acceptance word
          // only where some cell of the band may reject (else the particle ends at its first
          // candidate, so no later draw is taken)
          ub = all_real ? 0u : st.even_word();
          st.j += 2;
          f.D = __fmul_rn(-__logf(word_uniform<float>(st.first)), vtm);
          cnt.v[CNT_FLIGHTS] += 1;
          const unsigned qwx = (unsigned)((yg ? f.s1 : f.s0) > 0 ? qw : -qw);
          // candidates (Sec. 3.2) until the particle collides for real or reaches a wall; a
          // decision within rounding of the FP64 walk's defers the particle to the FP64 replay
          const int m0 = faces_to_wall(f.i0, f.s0, n0), m1 = faces_to_wall(f.i1, f.s1, n1);
          float eD = fmaf(f.D, TIE_LOG_REL, ea);  // bound of |D - D_fp64|
          bool wall_exit = false, deferred = false;
          int fb0 = 0, fb1 = 0;  // faces before the latest candidate, per axis
          int kc = 0;            // candidates tallied
#pragma unroll 1
          for (;;) {
            const float base = fmaf(TIE_REL, f.D, eD);
            if (f.D - f.tex > base) {
              wall_exit = true;
              break;
            }
            if (f.tex - f.D <= fmaf(TIE_REL, f.tex, eD)) {  // at the first wall within rounding
              deferred = true;
              break;
            }
            bool near = false;  // a count within the bound of a face, found with it for all-real bands
            if (all_real) {
              fb0 = count_near(f.D, f.t0, f.d0, base, near);
              fb1 = count_near(f.D, f.t1, f.d1, base, near);
            } else {
              fb0 = faces_before(f.D, f.t0, f.d0);
              fb1 = faces_before(f.D, f.t1, f.d1);
            }
            const int cell = clampi(f.i0 + f.s0 * fb0, n0) + n0 * clampi(f.i1 + f.s1 * fb1, n1);
            const long long ci = bcbase + cell;
            const int oc = candidate_outcome<2>(A, bcbase, ncells, f, base, fb0, fb1, 0, cell, all_real, near, ub,
                                                n0, n1, 1, n0, 0);
            if (oc == CAND_DEFER) {
              deferred = true;
              break;
            }
            cnt.v[CNT_CANDIDATES] += 1;
            ++kc;
            if (!all_real) {  // else W = tau_maj R after the sweep
              if (K32 && S.W32) tally_k32(&S.W32[ci], w);
              else if (!K32 && A.W) atomicAdd(&A.W[ci], w);
            }
            if (oc == CAND_REAL) {
              cnt.v[CNT_REAL] += 1;
              if (K32) tally_k32(&S.R32[ci], w);
              else atomicAdd(&A.R[ci], w);
              if (yg) atomicAdd(&S.DY[coff + cell], w);
              break;
            }
            uint32_t uw;
            st.next_pair(uw, ub);
            const float ell = __fmul_rn(-__logf(word_uniform<float>(uw)), vtm);
            f.D = __fadd_rn(f.D, ell);
            eD = fmaf(f.D, TIE_SUM, fmaf(ell, TIE_LOG_REL, eD + ea));
          }
          // faces crossed before the end per axis: at a real collision those before its
          // candidate; at a wall the exit axis's count is known and the other axis's follows
          // from the exit distance (within rounding of one of its faces, near a cell corner,
          // the particle is deferred too)
          int ex = -1, c0, c1;
          if (wall_exit) {
            // the face count of the axis not exited, near a cell corner within rounding of
            // the FP64 walk's: deferred too
            const float bx = TIE_REL * f.tex;
            ex = f.i2;
            const int q = count_near(f.tex, ex == 0 ? f.t1 : f.t0, ex == 0 ? f.d1 : f.d0, bx, deferred);
            c0 = ex == 0 ? m0 - 1 : min(q, m0 - 1);
            c1 = ex == 1 ? m1 - 1 : min(q, m1 - 1);
          } else {
            c0 = min(fb0, m0 - 1);
            c1 = min(fb1, m1 - 1);
          }
          if (deferred) {
            defer_particle(S, G.first + (unsigned)q * (unsigned)G.ne + (unsigned)rank, ((unsigned)kc << 1) | (yg ? 1u : 0u));
          } else {
            if (wall_exit) cnt.v[CNT_WALL_EXITS] += 1;
            cnt.v[CNT_CROSSINGS] += c0 + c1;
            // face items along the tallied axis p: a0 + k sp + sq min(ceil(u0 + k r), lim)
            // p: the tallied axis (x for the x-group), q: the other one; selects, no branch
            const float tp = yg ? f.t1 : f.t0, tq = yg ? f.t0 : f.t1;
            const float dp = yg ? f.d1 : f.d0, dq = yg ? f.d0 : f.d1;
            const int cp = yg ? c1 : c0, mq = yg ? m0 : m1, axp = yg ? 1 : 0;
            if (ex == 1 - axp && (yg ? f.s0 : f.s1) < 0) {  // exit through the low q-wall
              const int j = yg ? in.wface_off[0] + f.i1 + f.s1 * c1 : in.wface_off[2] + f.i0 + f.s0 * c0;
              atomicAdd(&gx[j], -w);
            }
            nitem = cp + (ex == axp ? 1 : 0);
            const bool flat = !(dq < INFINITY);
            const float u0 = flat ? -1.f : __fdividef(tp - tq, dq);
            const float r = flat ? 0.f : __fdividef(dp, dq);
            const int lim = mq - 1;
            const int a0 = yg ? (int)fax1 + f.i0 + n0 * (f.i1 + (f.s1 > 0 ? 1 : 0))
                              : f.i0 + (f.s0 > 0 ? 1 : 0) + sy_xf * f.i1;
            const int sp = yg ? f.s1 * n0 : f.s0;
            const int sq = yg ? f.s0 : f.s1 * sy_xf;
            // (a count's bits come with those of 2^23: the first face takes them out)
            pa_own = make_int4((int)((unsigned)(a0 - wbase) - (unsigned)sq * 0x4B000000u), sp, sq, lim + 0x4B000000);
            pb_own = make_int4(__float_as_int(u0), __float_as_int(r), (int)qwx, 0);
          }
        }
      // ---- the pass's face items: each lane's list is cut into segments of SEG items, the
      // segments are numbered in lane order and dealt to the lanes round-robin, 32 to a
      // round; a lane runs SEG steps of its segment with its list's parameters (no per-item
      // list check). Against contiguous chunks of the pass's items (a list change inside a
      // chunk at a different step on every lane): 2.46 -> 2.40 ms per bench-batch sweep (Kn
      // 10: -6 %, Kn 0.01, short lists: +3 %). The non-empty lists are stored in lane order
      // without gaps; segment g belongs to list (number of lists starting at or before g) - 1,
      // counted from a ballot of the lists starting before the round and an OR-reduction of
      // the start bits within it (no search through the starts in shared memory). ----
      constexpr int SEG = 8;
      const int nseg = (nitem + SEG - 1) / SEG;
      int incl = nseg;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      const int total = __shfl_sync(0xffffffffu, incl, 31);
      if (total > 0) {
        const int first = incl - nseg;  // this lane's first segment
        const unsigned nonempty = __ballot_sync(0xffffffffu, nseg > 0);
        if (nseg > 0) {
          const int pos = __popc(nonempty & ((1u << lane) - 1u));
          lst[pos] = first;
          par[2 * pos] = pa_own;
          par[2 * pos + 1] = make_int4(pb_own.x, pb_own.y, pb_own.z, nitem);
        }
        __syncwarp();
        for (int r0 = 0; r0 < total; r0 += 32) {
          const bool starts_here = nseg > 0 && first >= r0 && first < r0 + 32;
          const unsigned bits = __reduce_or_sync(0xffffffffu, starts_here ? 1u << (first - r0) : 0u);
          const int before = __popc(__ballot_sync(0xffffffffu, nseg > 0 && first < r0));
          const int g = r0 + lane;
          if (g >= total) continue;
          const int l = before + __popc(bits & (0xffffffffu >> (31 - lane))) - 1;
          const int4 pa = par[2 * l], pb = par[2 * l + 1];
          const int kl0 = (g - lst[l]) * SEG;
          const int kn = min(SEG, pb.w - kl0);
          const float fk0 = small_int_float(kl0), r = __int_as_float(pb.y), u0 = __int_as_float(pb.x);
          const unsigned q = (unsigned)pb.z;
          unsigned at = (unsigned)pa.x + (unsigned)kl0 * (unsigned)pa.y;
#pragma unroll
          for (int t = 0; t < SEG; ++t, at += (unsigned)pa.y) {
            if (t >= kn) break;
            // item kl0 + t: its row (column), min(ceil(max(u0 + k r, 0)), lim), in the low bits of a
            // sum rounded upwards (this loop issues a third of the kernel's instructions at 34 faces
            // a flight; without the conversions and the subtraction of the bits of 2^23 per item the
            // cavity batch takes 1904 us per sweep, with them 1966)
            const float c = __fadd_ru(fmaxf(fmaf(fk0 + (float)t, r, u0), 0.f), 8388608.f);
            const unsigned rel = at + (unsigned)pa.z * (unsigned)min(__float_as_int(c), pa.w);
            if (PARTIAL && rel >= wlen) {  // outside the window: the same contribution, globally
              add_units(S.Fi, face_off + wbase + (int)rel, (long long)(int)q);
              continue;
            }
            const unsigned old = atomicAdd(&win[rel], q);
            // |q| <= 2^26, so the word can wrap only from within 2^26 of 0 / 2^32
            if (old + 0x04000000u < 0x08000000u) {
              const int carry = ((int)q >> 31) + (old + q < old ? 1 : 0);
              if (carry) add_units(S.Fi, face_off + wbase + (int)rel, (long long)carry << 32);
            }
          }
        }
        __syncwarp();
      }
      }
      if (n_yg > 0) {
        if (kind == 0) {
          atomicAdd(&S.DY[coff + e], -(double)n_yg * w);
        } else {
          const int wl = kind - 1;
          atomicAdd(&S.EY[in.bface_off + in.wface_off[wl] + e], (double)n_yg * ((wl & 1) ? -w : w));
        }
      }
    }
    __syncthreads();
    for (unsigned i = threadIdx.x; i < wlen; i += STAGED_NT) {
      const int v = (int)(win[i] - WIN_BIAS);
      if (v) add_units(S.Fi, face_off + wbase + i, v);
    }
    __syncthreads();
  }
  flush_lcounts(cnt, A.counters);
}

template <bool K32>
void launch_sync(const Ctx* c, const SweepArgs& a, const StagedArgs& S, int blocks, size_t smem, cudaStream_t s) {
  SyncArgs Y;
  Y.L.groups = c->d_sync_groups;
  Y.L.n_groups = a.n_groups;
  Y.L.n_tasks = c->sync_tasks;
  Y.L.qch = c->sync_qch;
  Y.L.next = nullptr;
  Y.L.lamVm = nullptr;
  Y.L.max_j = 0;
  Y.task_end = c->d_sync_end;
  if (c->all_real_all) {
    if (c->sync_partial) sweep_sync_kernel<K32, true, true><<<blocks, STAGED_NT, smem, s>>>(a, S, Y);
    else sweep_sync_kernel<K32, true, false><<<blocks, STAGED_NT, smem, s>>>(a, S, Y);
  } else {
    if (c->sync_partial) sweep_sync_kernel<K32, false, true><<<blocks, STAGED_NT, smem, s>>>(a, S, Y);
    else sweep_sync_kernel<K32, false, false><<<blocks, STAGED_NT, smem, s>>>(a, S, Y);
  }
}

cudaError_t launch_sweep_staged(const Ctx* c, const SweepArgs& a_in, cudaStream_t s) {
  // 1D and 2D: the trace's fixed-point face sums go to Fi, the FP64 ones to Fx, and the closing
  // pass writes every face of the caller's F from them; 3D tallies in the caller's F directly
  SweepArgs a = a_in;
  const bool fixed = a_in.F && c->dim <= 2;
  if (fixed) a.F = c->d_Fx;
  StagedArgs S = {};
  S.n_inst = c->n_inst;
  S.inst_next = c->d_inst_next;
  S.inst_end = c->d_inst_end;
  S.cost_prefix = c->d_cost_prefix;
  S.cost_total = c->cost_total;
  S.window = c->d_window;
  S.wmax = reinterpret_cast<const double*>(c->d_wmax);
  S.warp_grab = c->opt.warp_grab > 0 ? c->opt.warp_grab : 256;
  S.walk_k = c->opt.walk_k > 0 ? c->opt.walk_k : 16;
  S.refill = c->opt.refill_lanes;
  S.group_mag = c->d_group_mag;
  S.mag_n0 = c->d_mag;
  S.mag_n1 = c->d_mag + c->n_inst;
  S.mag_wall = c->d_mag + 2 * c->n_inst;
  S.defer = c->d_defer;
  S.defer_n = c->d_defer_n;
  S.defer_cap = c->defer_cap;
  S.err = c->d_err;
  S.DY = c->d_DY;
  S.EY = c->d_EY;
  S.GX = c->d_GX;
  S.gx_stride = c->total_bfaces;
  S.Fi = c->d_Fi;
  const bool k32 = c->opt.tally == IUGKP_TALLY_STAGED_K32;
  const size_t bc = (size_t)c->nb * c->total_cells;
  S.R32 = k32 ? c->d_R32 : nullptr;
  S.W32 = k32 && a.W ? c->d_W32 : nullptr;
  S.F32 = k32 && a.F ? c->d_F32 : nullptr;
  const bool sync = sync_schedule(c) && a.F;
  PrologueArgs P = {};
  auto clear = [&](void* p, size_t n) {
    if (!p || !n) return;
    P.clear[P.n_clear] = reinterpret_cast<unsigned long long*>(p);
    P.words[P.n_clear++] = (long long)n;
  };
  if (k32) {
    clear(S.R32, bc);
    clear(S.W32, bc);
    clear(S.F32, (size_t)c->total_faces);
  } else {
    clear(a.R, bc);
    if (!c->all_real_all) clear(a.W, bc);  // else W = tau_maj R afterwards
  }
  if (a.F) clear(a.F, (size_t)c->total_faces);
  if (fixed) clear(c->d_Fi, (size_t)c->total_faces);
  if (a.F && c->dim == 2) {
    clear(c->d_GX, (size_t)GX_COPIES * c->total_bfaces);
    if (c->any_two_group) {
      clear(c->d_DY, (size_t)c->total_cells);
      clear(c->d_EY, (size_t)c->total_bfaces);
    }
  }
  clear(a.counters, CNT_N);
  clear(c->d_defer_n, 2);
  P.n_inst = c->n_inst;
  P.next = c->d_inst_next;
  P.next_from = sync ? c->d_sync_beg : c->d_inst_beg;
  P.wmax_blocks = c->wmax_blocks;
  P.bpre = c->d_wmax_bpre;
  P.wpart = c->d_wpart;
  P.wmax = c->d_wmax;
  P.ticket = c->d_ticket;
  cudaError_t e = launch_prologue(c, a, P, s);
  if (e != cudaSuccess) return e;
  const size_t smem = (size_t)c->staged_cap * sizeof(unsigned);
  const int blocks = c->sm_count * c->staged_blocks_per_sm;
  if (k32) {
    switch (c->dim) {
      case 1: sweep_staged_kernel<1, true><<<blocks, STAGED_NT, smem, s>>>(a, S); break;
      case 2:
        if (sync) launch_sync<true>(c, a, S, blocks, smem, s);
        else sweep_staged_kernel<2, true><<<blocks, STAGED_NT, smem, s>>>(a, S);
        break;
      default: launch_chain(c, a, S, true, s); break;
    }
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    const int fb = c->sm_count * 4;
    k32_finalize_kernel<<<fb, 256, 0, s>>>(c->d_R32, a.R, (long long)bc, 0);
    if (a.W) k32_finalize_kernel<<<fb, 256, 0, s>>>(c->d_W32, a.W, (long long)bc, 0);
    if (a.F && (c->dim == 3 || !sync)) k32_finalize_kernel<<<fb, 256, 0, s>>>(c->d_F32, a.F, c->total_faces, 1);
    // the deferred particles add to the FP64 outputs (after the finalize, which overwrites R and W)
  } else {
    switch (c->dim) {
      case 1: sweep_staged_kernel<1, false><<<blocks, STAGED_NT, smem, s>>>(a, S); break;
      case 2:
        if (sync) launch_sync<false>(c, a, S, blocks, smem, s);
        else sweep_staged_kernel<2, false><<<blocks, STAGED_NT, smem, s>>>(a, S);
        break;
      default: launch_chain(c, a, S, false, s); break;
    }
  }
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = launch_replay(c, a, S, s)) != cudaSuccess) return e;
  if (c->dim == 3) return launch_close_3d(c, a_in, s);
  if (c->dim == 2) return launch_close_2d(c, a_in, s);
  return launch_close_1d(c, a_in, s);
}

cudaError_t launch_k32_finalize(const Ctx* c, const float2* src, double* dst, long long n, cudaStream_t s) {
  k32_finalize_kernel<<<c->sm_count * 4, 256, 0, s>>>(src, dst, n, 0);
  return cudaGetLastError();
}

// Measured accuracy of the FP32 operations the tie bounds rely on, over every uniform the
// walk can draw ((2m + 1) 2^-24, m < 2^23), against FP64:
//  out[0] max |__logf(u) - ln u| / (TIE_LOG_ABS + (TIE_LOG_REL - 2^-23) |ln u|) (the log's
//         share of the bound on a flight length; <= 1 required);
//  out[1] max relative error of sincospif(2u), both outputs, in units of 2^-23;
//  out[2] max relative error of sqrtf(fmaf(-mu, mu, 1)), mu = 2u - 1, units of 2^-23;
//  out[3] max relative error of sqrtf(u) and sqrtf(1 - u), units of 2^-23;
//  out[4] max relative error of __fdividef(x, y) over pairs of uniforms, units of 2^-23.
// Results are max-reduced as the bit patterns of non-negative doubles.
__global__ void walk_bounds_kernel(unsigned long long* out) {
  double e[5] = {0, 0, 0, 0, 0};
  for (unsigned m = blockIdx.x * blockDim.x + threadIdx.x; m < (1u << 23); m += gridDim.x * blockDim.x) {
    const float u = word_uniform<float>(m << 9);
    const double ud = (double)u;
    const double lg = log(ud);
    e[0] = fmax(e[0], fabs((double)__logf(u) - lg) / ((double)TIE_LOG_ABS + ((double)TIE_LOG_REL - 0x1p-23) * fabs(lg)));
    float sp, cp;
    sincospif(2.f * u, &sp, &cp);
    double sd, cd;
    sincospi(2.0 * ud, &sd, &cd);
    e[1] = fmax(e[1], fmax(fabs(sp - sd) / fabs(sd), fabs(cp - cd) / fabs(cd)) * 0x1p23);
    const float mu = 2.f * u - 1.f;
    const double sn = sqrt(1.0 - (double)mu * (double)mu);
    e[2] = fmax(e[2], fabs((double)sqrtf(fmaf(-mu, mu, 1.f)) - sn) / sn * 0x1p23);
    e[3] = fmax(e[3], fmax(fabs((double)sqrtf(u) - sqrt(ud)) / sqrt(ud),
                           fabs((double)sqrtf(1.f - u) - sqrt(1.0 - ud)) / sqrt(1.0 - ud)) * 0x1p23);
    // pairs (u, u') with u' another uniform, the divisor scaled over several binades
    const float v = word_uniform<float>((m * 2654435761u) << 9) * __int_as_float((127 - (int)(m & 15u)) << 23);
    const double q = ud / (double)v;
    e[4] = fmax(e[4], fabs((double)__fdividef(u, v) - q) / q * 0x1p23);
  }
  for (int k = 0; k < 5; ++k) {
    double x = e[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_down_sync(0xffffffffu, x, o));
    if ((threadIdx.x & 31) == 0) atomicMax(&out[k], (unsigned long long)__double_as_longlong(x));
  }
}

cudaError_t launch_walk_bounds(unsigned long long* out, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(out, 0, 5 * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  walk_bounds_kernel<<<1024, 256, 0, s>>>(out);
  return cudaGetLastError();
}

// FP64 atomic additions to scattered addresses of an L2-resident array (the deposit tallies'
// access pattern): every thread adds to `per_thread` addresses spread by a multiplicative hash.
__global__ void atomic_rate_kernel(double* buf, unsigned mask, int per_thread) {
  const unsigned t = blockIdx.x * blockDim.x + threadIdx.x;
  for (int k = 0; k < per_thread; ++k) {
    const unsigned a = ((t * 32u + (unsigned)k) * 2654435761u) & mask;
    atomicAdd(&buf[a], 1.0);
  }
}

cudaError_t measure_atomic_rate(int sm_count, double* out_rate) {
  const unsigned n = 1u << 20;  // 8 MB: L2-resident
  double* buf = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaError_t e = cudaMalloc((void**)&buf, n * sizeof(double));
  if (e == cudaSuccess) e = cudaMemset(buf, 0, n * sizeof(double));
  if (e == cudaSuccess) e = cudaEventCreate(&e0);
  if (e == cudaSuccess) e = cudaEventCreate(&e1);
  const int blocks = sm_count * 8, threads = 256, per = 256;
  float ms = 0.f;
  if (e == cudaSuccess) {
    atomic_rate_kernel<<<blocks, threads>>>(buf, n - 1, per);  // warm-up
    cudaEventRecord(e0);
    for (int r = 0; r < 5; ++r) atomic_rate_kernel<<<blocks, threads>>>(buf, n - 1, per);
    cudaEventRecord(e1);
    e = cudaEventSynchronize(e1);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
  }
  if (e == cudaSuccess) *out_rate = 5.0 * blocks * threads * (double)per / (ms * 1e-3);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  if (buf) cudaFree(buf);
  return e;
}

// The relative bound the face-count decision needs, from the measured errors above (units of
// 2^-23): direction s = product of a square root and a sine/cosine (one more rounding), cell
// size h in FP32 (half an ulp), d = h / |s| (__fdividef), t = (1 - xi) d (one rounding), the
// quotient (D - t) / d (__fdividef) and the difference D - t (half an ulp each), and half an
// ulp for the distance to the face. Returned as a fraction of TIE_REL (<= 1 required).
double walk_bound_fraction(const double* m) {
  const double ulp = 0x1p-23;
  const double Es = (std::max(m[2], m[3]) + m[1] + 0.5) * ulp;
  const double Ed = 0.5 * ulp + Es + m[4] * ulp;
  const double Et = Ed + 0.5 * ulp;
  return (Et + Ed + m[4] * ulp + ulp) / (double)TIE_REL;
}

cudaError_t allow_shared(const void* kernel, size_t optin) {
  cudaFuncAttributes at;
  const cudaError_t e = cudaFuncGetAttributes(&at, kernel);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(optin - at.sharedSizeBytes));
}

cudaError_t configure_staged(Ctx* c) {
  cudaError_t e = cudaSuccess;
  if (c->dim == 3) return configure_chain(c);
  const size_t smem = (size_t)c->staged_cap * sizeof(unsigned);
  const void* fwd[4] = {(const void*)sweep_staged_kernel<1, false>, (const void*)sweep_staged_kernel<2, false>,
                        (const void*)sweep_staged_kernel<1, true>, (const void*)sweep_staged_kernel<2, true>};
  for (const void* f : fwd)
    if ((e = allow_shared(f, c->smem_optin)) != cudaSuccess) return e;
  const void* syn[8] = {(const void*)sweep_sync_kernel<false, false, false>, (const void*)sweep_sync_kernel<true, false, false>,
                        (const void*)sweep_sync_kernel<false, true, false>, (const void*)sweep_sync_kernel<true, true, false>,
                        (const void*)sweep_sync_kernel<false, false, true>, (const void*)sweep_sync_kernel<true, false, true>,
                        (const void*)sweep_sync_kernel<false, true, true>, (const void*)sweep_sync_kernel<true, true, true>};
  for (const void* f : syn)
    if ((e = allow_shared(f, c->smem_optin)) != cudaSuccess) return e;
  int nb = 0, nk = 0;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fwd[c->dim - 1], STAGED_NT, smem)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nk, fwd[c->dim + 1], STAGED_NT, smem)) != cudaSuccess) return e;
  nb = std::min(nb, nk);  // one grid size for both tally modes
  c->staged_blocks_per_sm = nb > 0 ? nb : 1;
  return cudaSuccess;
}

}  // namespace iugkp
