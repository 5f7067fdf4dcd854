// Forward sweep kernels: emission, cell-by-cell walk, null collisions and tallies.
// arXiv 2506.09465 Sec. 3.1 (steps (1)-(3)) and Sec. 3.2 (steps (1)-(6), with the
// candidate chain of a particle completed inside one sweep).
#include <cuda_runtime.h>

#include "device.cuh"
#include "internal.h"
#include "plain.cuh"
#include "replay.cuh"

namespace iugkp {

// Tallies of the plain sweep: every candidate, real collision, face and wall, each a global
// FP64 atomic.
struct PlainTally {
  const SweepArgs& A;
  const InstDesc& in;
  double w, wt;  // weight; weight x tau_maj (the candidate estimator W)
  __device__ bool candidate(int, long long ci) {
    if (A.W) atomicAdd(&A.W[ci], wt);
    return true;
  }
  __device__ void real(long long ci, int) { atomicAdd(&A.R[ci], w); }
  __device__ void cross(int, int stp, long long face) {
    if (A.F) atomicAdd(&A.F[in.face_off + face], stp > 0 ? w : -w);
  }
  __device__ void exit(int a, int stp, long long) {
    if (A.wall) atomicAdd(&A.wall[in.wall_off + 2 * a + (stp > 0 ? 1 : 0)], w);
  }
};

// One particle from emission to absorption (one thread, global FP64 atomics).
template <typename Real, int DIM>
__device__ __forceinline__ void run_particle(const SweepArgs& A, long long pid, Counts& cnt) {
  int gi;
  double w;
  Walk<Real, DIM> wk;
  Stream st;
  if (!emit_particle<Real, DIM>(A, pid, gi, w, wk, st)) return;
  const Group G = A.groups[gi];
  const InstDesc& in = A.inst[G.inst];
  cnt.v[CNT_FLIGHTS] += 1;
  PlainTally pol{A, in, w, w * A.taumaj[(long long)G.inst * A.nb + G.band]};
  walk_particle<Real, DIM>(A, in, G.inst, G.band, wk, st, cnt, pol);
}

// Deposit tallies of a replayed particle: W as w (the staged sweep scales it by tau_maj
// afterwards, or sets it to tau_maj R in bands whose every candidate is real: all_real), from
// candidate k_done on (the earlier ones were tallied by the staged sweep); R, and the y-group
// balance DY for a y-group particle of a two-group instance.
struct ReplayDeposits {
  const SweepArgs& A;
  const StagedArgs& S;
  const InstDesc& in;
  double w;
  int k_done;
  bool ydy;
  bool all_real;
  Counts& cnt;
  __device__ void candidate(int k, long long ci, int) {
    if (k < k_done) return;
    cnt.v[CNT_CANDIDATES] += 1;
    if (A.W && !all_real) atomicAdd(&A.W[ci], w);
  }
  __device__ void real(long long ci, int cell) {
    cnt.v[CNT_REAL] += 1;
    atomicAdd(&A.R[ci], w);
    if (ydy) atomicAdd(&S.DY[in.cell_off + cell], w);
  }
};

// Face index within the instance of face coordinate f along axis a, cell coordinates c[] on
// the other axes.
__device__ __forceinline__ long long face_at(const InstDesc& in, int a, int f, const int* c) {
  if (a == 0) return in.fax_off[0] + f + (long long)(in.n[0] + 1) * (c[1] + (long long)in.n[1] * c[2]);
  if (a == 1) return in.fax_off[1] + c[0] + (long long)in.n[0] * (f + (long long)(in.n[1] + 1) * c[2]);
  return in.fax_off[2] + c[0] + (long long)in.n[0] * (c[1] + (long long)in.n[1] * f);
}

__device__ __forceinline__ double shfl_d(double x, int src) {
  return __hiloint2double(__shfl_sync(0xffffffffu, __double2hiint(x), src),
                          __shfl_sync(0xffffffffu, __double2loint(x), src));
}

// The real collision of a landing sweep's particle (forward index pid, nothing tallied yet) in FP64.
template <int DIM>
__device__ __forceinline__ void replay_real(const SweepArgs& A, const StagedArgs& S, unsigned pid) {
  Counts cnt;  // a landing sweep's event counts are not read
  const Group G = A.groups[find_group(A.groups, A.n_groups, (long long)pid)];
  const InstDesc& in = A.inst[G.inst];
  const unsigned local = pid - (unsigned)G.first_particle;
  const int q = (int)(local / (unsigned)G.n_emitters);
  int e = (int)(local - (unsigned)q * (unsigned)G.n_emitters);
  if (G.perm_off >= 0) e = A.perm[G.perm_off + e];  // the staged visiting order
  int gj, fb[DIM];
  double w;
  Walk<double, DIM> wk;
  Stream st;
  if (!emit_particle<double, DIM, false>(A, G.first_particle + (long long)e * G.per_emitter + q, gj, w, wk, st)) return;
  Seg64<DIM> sg;
  sg.init(wk, in);
  ReplayDeposits pol{A, S, in, w, 0, false, false, cnt};
  if (replay_candidates<DIM>(A, in, G.inst, G.band, wk, sg, st, fb, pol) < 0) atomicOr(A.err, ERR_BUDGET);
}

// One thread per queue entry follows the particle's candidates in FP64 and makes its deposit
// tallies; then the warp tallies the face items of its particles together, one particle at a
// time (its segment broadcast from its lane), the lanes taking successive items. Faces
// tallied: those the staged sweep tallies for this particle (x in 1D; x and y in 3D; x in 2D,
// or y for a y-group particle of a two-group instance), the wall faces among them included;
// an exit through the low wall of an untallied axis goes to that wall's face (one-group
// instances) or to the group's exit tally GX (two-group). Emission needs nothing: the staged
// sweep and its post-passes account for it.
// LAND: after a landing sweep, whose particles beyond the queue follow (the full sweeps keep the kernel
// without them: its stack is half as deep).
template <int DIM, bool LAND>
__global__ void __launch_bounds__(256) replay_kernel(SweepArgs A, StagedArgs S) {
  Counts cnt;
#pragma unroll
  for (int k = 0; k < CNT_N; ++k) cnt.v[k] = 0;
  const int lane = threadIdx.x & 31;
  const unsigned n = min(*S.defer_n, S.defer_cap);
  // Warp j of block b is warp a = j G + b (G blocks: warp j of every block comes before warp
  // j + 1 of any), and warp a takes entries E a .. E a + E - 1 (then E (a + W) .., W warps in the
  // grid). The queue is short: numbered b 8 + j, the warps that got work were all in the first
  // few blocks, on a few SMs (measured: the busiest SM active 3.6 times as long as the average);
  // this way the first warps to get work are the first warp of every block. E, at most 32, is
  // what spreads the queue over G / 2 warps (four per SM): a warp's particles share its FP64
  // instructions, but their faces are tallied one particle after the other, so a queue of a few
  // hundred is done sooner with one or two particles per warp.
  const unsigned W = gridDim.x * blockDim.x >> 5;
  const unsigned wid = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const unsigned half = max(1u, gridDim.x >> 1), E = min(32u, max(1u, (n + half - 1) / half));
  // all lanes of a warp run the same rounds (the face items are tallied by the whole warp)
  for (unsigned i0 = E * wid; i0 < n; i0 += E * W) {
    const unsigned i = lane < (int)E ? i0 + lane : n;
    // the lane's particle, kept for the face items
    int kinst = 0, ex = 0, tall = 0;  // instance, exit axis (-1: real collision), tallied axes (bits)
    double w = 0.0;
    double t[3] = {0, 0, 0}, d[3] = {0, 0, 0}, id[3] = {0, 0, 0};
    int idx[3] = {0, 0, 0}, step[3] = {1, 1, 1}, m[3] = {1, 1, 1}, items[3] = {0, 0, 0};
    if (i < n) {
      const uint2 ent = S.defer[i];
      const Group G = A.groups[find_group(A.groups, A.n_groups, (long long)ent.x)];
      const InstDesc& in = A.inst[G.inst];
      const unsigned local = ent.x - (unsigned)G.first_particle;
      const int q = (int)(local / (unsigned)G.n_emitters);
      int e = (int)(local - (unsigned)q * (unsigned)G.n_emitters);
      if (G.perm_off >= 0) e = A.perm[G.perm_off + e];  // the staged visiting order
      int gj;
      Walk<double, DIM> wk;
      Stream st;
      if (emit_particle<double, DIM, false>(A, G.first_particle + (long long)e * G.per_emitter + q, gj, w, wk, st)) {
        Seg64<DIM> sg;
        sg.init(wk, in);
        const bool two = DIM == 2 && A.F && S.window[G.inst].x == 0 && (long long)S.window[G.inst].y == in.nfaces;
        const bool yg = two && (ent.y & 1u);
        ReplayDeposits pol{A, S, in, w, (int)(ent.y >> 1), yg,
                           A.all_real[(long long)G.inst * A.nb + G.band] != 0, cnt};
        int fb[DIM];
        const int res = replay_candidates<DIM>(A, in, G.inst, G.band, wk, sg, st, fb, pol);
        if (res < 0) {
          cnt.v[CNT_DROPPED] += 1;
          atomicOr(A.err, ERR_BUDGET);
        } else {
          // interior faces crossed per axis; at a wall the exit axis's are all of them
          const bool exit = res == 0;
          int c[3] = {0, 0, 0};
#pragma unroll
          for (int a = 0; a < DIM; ++a) {
            c[a] = exit ? (a == sg.ex ? sg.m[a] - 1 : min(count_before64(sg.tex, sg.t[a], sg.id[a]), sg.m[a] - 1))
                        : fb[a];
            cnt.v[CNT_CROSSINGS] += c[a];
            t[a] = sg.t[a];
            d[a] = sg.d[a];
            id[a] = sg.id[a];
            idx[a] = wk.idx[a];
            step[a] = wk.step[a];
            m[a] = sg.m[a];
          }
          if (exit) cnt.v[CNT_WALL_EXITS] += 1;
          kinst = G.inst;
          ex = exit ? sg.ex : -1;
          if (A.F) {
#pragma unroll
            for (int a = 0; a < DIM; ++a) {
              const bool ta = DIM == 1 || (two ? a == (yg ? 1 : 0) : a < DIM - 1);
              if (ta) {
                tall |= 1 << a;
                items[a] = c[a] + (exit && sg.ex == a ? 1 : 0);
              }
            }
            if (exit && !((tall >> sg.ex) & 1) && wk.step[sg.ex] < 0) {
              // exit through the low wall of an untallied axis
              int cc[3] = {0, 0, 0};
#pragma unroll
              for (int a = 0; a < DIM; ++a) cc[a] = wk.idx[a] + wk.step[a] * c[a];
              if (two) {
                const int j = sg.ex == 1 ? cc[0] : cc[1];  // the low y-wall's column or the low x-wall's row
                atomicAdd(&S.gx()[in.bface_off + in.wface_off[sg.ex == 1 ? 2 : 0] + j], -w);
              } else {
                atomicAdd(&A.F[in.face_off + face_at(in, sg.ex, 0, cc)], -w);
              }
            }
          }
        }
      }
    }
    // face items, particle by particle: item j along the tallied axis p is its j-th face, at
    // path length t_p + j d_p; the cell there on each other axis follows from its face count
    unsigned pend = __ballot_sync(0xffffffffu, tall != 0);
    while (pend) {
      const int src = __ffs(pend) - 1;
      pend &= pend - 1;
      const int k = __shfl_sync(0xffffffffu, kinst, src);
      const InstDesc& in = A.inst[k];
      const double ws = shfl_d(w, src);
      const int tl = __shfl_sync(0xffffffffu, tall, src);
      double ts[3], ds[3], is[3];
      int xs[3], ss[3], ms[3], ns[3];
#pragma unroll
      for (int a = 0; a < DIM; ++a) {
        ts[a] = shfl_d(t[a], src);
        ds[a] = shfl_d(d[a], src);
        is[a] = shfl_d(id[a], src);
        xs[a] = __shfl_sync(0xffffffffu, idx[a], src);
        ss[a] = __shfl_sync(0xffffffffu, step[a], src);
        ms[a] = __shfl_sync(0xffffffffu, m[a], src);
        ns[a] = __shfl_sync(0xffffffffu, items[a], src);
      }
#pragma unroll
      for (int p = 0; p < DIM; ++p) {
        if (!((tl >> p) & 1)) continue;
        const double sgn = ss[p] > 0 ? ws : -ws;
        for (int j = lane; j < ns[p]; j += 32) {
          const double T = ts[p] + (double)j * ds[p];
          int cc[3] = {0, 0, 0};
#pragma unroll
          for (int a = 0; a < DIM; ++a)
            if (a != p) cc[a] = xs[a] + ss[a] * min(count_before64(T, ts[a], is[a]), ms[a] - 1);
          const int f = ss[p] > 0 ? xs[p] + 1 + j : xs[p] - j;
          atomicAdd(&A.F[in.face_off + face_at(in, p, f, cc)], sgn);
        }
      }
    }
    (void)ex;
  }
  if (LAND) for_overflow(S, [&](unsigned pid) { replay_real<DIM>(A, S, pid); });
  flush_counts(cnt, A.counters);
}

template <bool LAND>
static void launch_replay_dim(const Ctx* c, const SweepArgs& a, const StagedArgs& S, cudaStream_t s) {
  const int blocks = c->sm_count * 8;
  switch (c->dim) {
    case 1: replay_kernel<1, LAND><<<blocks, 256, 0, s>>>(a, S); break;
    case 2: replay_kernel<2, LAND><<<blocks, 256, 0, s>>>(a, S); break;
    default: replay_kernel<3, LAND><<<blocks, 256, 0, s>>>(a, S); break;
  }
}

cudaError_t launch_replay(const Ctx* c, const SweepArgs& a, const StagedArgs& S, cudaStream_t s) {
  if (S.over) launch_replay_dim<true>(c, a, S, s);
  else launch_replay_dim<false>(c, a, S, s);
  return cudaGetLastError();
}

template <typename Real, int DIM>
__global__ void __launch_bounds__(256) sweep_plain_kernel(SweepArgs A) {
  Counts cnt;
#pragma unroll
  for (int k = 0; k < CNT_N; ++k) cnt.v[k] = 0;
  const long long nthreads = (long long)gridDim.x * blockDim.x;
  for (long long pid = (long long)blockIdx.x * blockDim.x + threadIdx.x; pid < A.total_particles; pid += nthreads)
    run_particle<Real, DIM>(A, pid, cnt);
  flush_counts(cnt, A.counters);
}

template <typename Real, int DIM>
static cudaError_t launch_plain(const Ctx* c, const SweepArgs& a, cudaStream_t s) {
  long long blocks = (a.total_particles + 255) / 256;
  long long cap = (long long)c->sm_count * 32;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  sweep_plain_kernel<Real, DIM><<<(unsigned)blocks, 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_sweep(const Ctx* c, const SweepArgs& a, cudaStream_t s) {
  const bool fp32 = c->opt.precision == IUGKP_TRACK_FP32;
  switch (c->dim) {
    case 1: return fp32 ? launch_plain<float, 1>(c, a, s) : launch_plain<double, 1>(c, a, s);
    case 2: return fp32 ? launch_plain<float, 2>(c, a, s) : launch_plain<double, 2>(c, a, s);
    default: return fp32 ? launch_plain<float, 3>(c, a, s) : launch_plain<double, 3>(c, a, s);
  }
}

}  // namespace iugkp
