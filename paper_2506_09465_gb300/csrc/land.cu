// Landing sweeps: the sweep where only the real collisions are asked for (R alone: the steady
// and averaging loops) and the adjoint re-trace. Same particles and draws as the staged sweep
// (sweep_staged.cu; arXiv 2506.09465 Sec. 3.1 steps (1)-(3), Sec. 3.2 null collisions).
// The cell of a candidate follows from its position along the segment (landing.cuh); nothing
// else is needed where no face is tallied: no distances to faces (one reciprocal and one
// quotient per axis), no counts, no exit.
#include <cuda_runtime.h>

#include <algorithm>

#include "device.cuh"
#include "internal.h"
#include "landing.cuh"
#include "staged.h"
#include "walk32.cuh"

namespace iugkp {

namespace {

template <bool K32>
__device__ __forceinline__ void deposit(const SweepArgs& A, const StagedArgs& S, long long j, double w) {
  if (K32) tally_k32(&S.R32[j], w);
  else atomicAdd(&A.R[j], w);
}

// Leaves a particle to the FP64 replay. The bound grows with the distance in cells: flights of some
// 10^4 cells leave more particles undecided (5 % of a film of 10^5 cells at Kn 1) than the queue
// holds (one in 32 and 65,536), and the plain FP64 kernel has no such limit; those beyond it are
// marked in a bitmap that the replay goes through. (Following them on the spot takes 120 registers
// in place of 64.)
__device__ __forceinline__ void land_defer(const StagedArgs& S, unsigned pid) {
  const unsigned i = atomicAdd(S.defer_n, 1u);
  if (i < S.defer_cap) S.defer[i] = make_uint2(pid, 0u);
  else atomicOr(&S.over[pid >> 5], 1u << (pid & 31u));
}

// Bands whose every candidate is real: one candidate per particle, no chain. A lane keeps its
// emitter for qch particles in a row (over its bands in turn: with tens of bands an emitter has
// only a few particles in each), so the cell coordinates, the weight, the first Philox rounds (the
// counter's emitter word does not change) and, in the adjoint, the gathered sum stay in registers;
// the lanes of a warp hold neighbouring emitters. Tasks (a tile of emitters x a run of particle
// numbers) are claimed one at a time by each warp.
template <int DIM, bool ADJ, bool K32>
__global__ void __launch_bounds__(LAND_NT) land_kernel(SweepArgs A, StagedArgs S, LandArgs L) {
  const int lane = threadIdx.x & 31;
  TaskGroup tg;
  for (;;) {
    unsigned task = 0;
    if (lane == 0) task = (unsigned)atomicAdd(L.next, 1ull);
    task = __shfl_sync(0xffffffffu, task, 0);
    if (task >= L.n_tasks) return;
    tg.find(L, task);
    int gi = tg.gi;
    const unsigned t = task - tg.t_beg;
    const int ntile = L.groups[gi].ntile, reps = L.groups[gi].reps, kind = L.groups[gi].kind;
    const int qc = (int)(t / (unsigned)ntile), tile = (int)(t - (unsigned)qc * (unsigned)ntile);
    int pass = qc * L.qch;
    const int pass_end = pass + L.qch;
    // the chain's first band with passes left
    while (L.groups[gi].next >= 0 && L.groups[L.groups[gi].next].pass0 <= pass) gi = L.groups[gi].next;
    const InstDesc& in = A.inst[L.groups[gi].inst];
    LaneEmitter<DIM> em;
    em.template init<ADJ>(A, S, L.groups[gi], in, tile, lane);
    const int n0 = in.n[0], n1 = in.n[1];
    const long long coff = in.cell_off;
    const uint32_t inst_id = in.inst_id;
    double gather = 0.0;
    for (;;) {
      const LandGroup& G = L.groups[gi];
      const int band = G.band, per = G.per, next = G.next;
      const unsigned first = G.first;
      const float vtm = A.vtm32[G.inst * A.nb + band], va = vtm * TIE_LOG_ABS;
      const long long bcbase = in.bc_off + (long long)band * in.ncells;
      const int band_end = next >= 0 ? min(pass_end, L.groups[next].pass0) : pass_end;
      double acc = 0.0;
      const int qend = em.on ? min(per, (band_end - G.pass0) * reps) : 0;
      for (int q = (pass - G.pass0) * reps + em.sub; q < qend; q += reps) {
        Stream st;
        st.init(A.seed, inst_id, (uint32_t)band, A.epoch, em.id, (uint32_t)q);
        float xi[3], s[3];
        emit_segment<DIM>(st, kind, xi, s);
        const float D = __fmul_rn(-__logf(word_uniform<float>(st.first)), vtm);
        const float eD = fmaf(D, TIE_LOG_REL, va), rel = fmaf(D, LAND_REL, eD);
        bool out = false, near = false;
        int o[3] = {0, 0, 0};
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
          const float g = s[a] * em.ih[a];
          const float X = fmaf(g, D, xi[a]), tol = fmaf(fabsf(g), rel, LAND_ABS);
          out |= em.lo[a] - X > tol || X - em.hi[a] > tol;  // beyond a wall for the FP64 walk too
          o[a] = floor_near(X, tol, near);
        }
        if (out) continue;
        if (near) {
          land_defer(S, first + (unsigned)q * (unsigned)L.groups[gi].ne + (unsigned)em.rank);
          continue;
        }
        const int cell = em.cell0 + o[0] + (DIM >= 2 ? n0 * o[1] : 0) + (DIM == 3 ? n0 * n1 * o[2] : 0);
        if (ADJ) acc += L.lamVm[coff + cell];
        else deposit<K32>(A, S, bcbase + cell, em.w);
      }
      if (ADJ && em.on) gather = fma(acc, em.w, gather);
      pass = band_end;
      if (next < 0 || pass >= pass_end) break;
      gi = next;
      em.template weight<ADJ>(A, L.groups[gi], in);
    }
    if (ADJ) {
      if (kind == 0) {
        if (gather != 0.0) atomicAdd(&A.adj_out[coff + em.e], gather);
      } else {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) gather += __shfl_down_sync(0xffffffffu, gather, d);
        if (lane == 0 && gather != 0.0) atomicAdd(&A.adj_wall[in.wall_off + kind - 1], gather);
      }
    }
  }
}

// Bands with null candidates: every lane follows the candidates of its own particle, and a warp
// refills its idle lanes once LAND_REFILL of them are idle (particles q-major in the group's
// visiting order, claimed in runs, as in sweep_staged_kernel).
template <int DIM, bool ADJ, bool K32>
__global__ void __launch_bounds__(LAND_NT) land_chain_kernel(SweepArgs A, StagedArgs S, LandArgs L) {
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u, total = (unsigned)A.total_particles;
  unsigned rbeg = 0, rend = 0, pid = 0;
  bool alive = false, exhausted = false;
  unsigned g_first = 1, g_end = 0, g_mag = 0;  // the lane's cached group
  int g_ne = 1, g_perm = -1, kind = 0, band = 0, inst = 0, emitter = 0, acc_slot = 0, acc_inst = 0;
  bool all_real = false;
  long long bcbase = 0, coff = 0;
  int n0 = 1, n1 = 1, n2 = 1, cell0 = 0;
  float vtm = 0.f, D = 0.f, eD = 0.f;
  float xi[3], g[3], lo[3], hi[3];
  uint32_t ub = 0;
  double w = 0.0, acc = 0.0;
  Stream st;
  auto flush_wall = [&] {
    if (acc != 0.0) atomicAdd(&A.adj_wall[A.inst[acc_inst].wall_off + acc_slot], acc);
    acc = 0.0;
  };
  for (;;) {
    const unsigned dead = __ballot_sync(0xffffffffu, !alive);
    if (!exhausted && (__popc(dead) >= LAND_REFILL)) {
      if (rbeg == rend) {
        unsigned long long got = 0;
        if (lane == 0) got = atomicAdd(L.next, (unsigned long long)S.warp_grab);
        got = __shfl_sync(0xffffffffu, got, 0);
        if (got < total) {
          rbeg = (unsigned)got;
          rend = (unsigned)min(got + (unsigned long long)S.warp_grab, (unsigned long long)total);
        } else {
          exhausted = true;
        }
      }
      const unsigned r = __popc(dead & lt_mask), take = min((unsigned)__popc(dead), rend - rbeg);
      if (!alive && r < take) {
        pid = rbeg + r;
        if (pid < g_first || pid >= g_end) {
          const int gi = find_group(A.groups, A.n_groups, (long long)pid);
          const Group G = A.groups[gi];
          g_first = (unsigned)G.first_particle;
          g_end = (unsigned)(G.first_particle + (long long)G.n_emitters * G.per_emitter);
          g_ne = G.n_emitters;
          g_mag = S.group_mag[gi];
          g_perm = G.perm_off;
          kind = G.kind;
          band = G.band;
          inst = G.inst;
          const InstDesc& in = A.inst[inst];
          n0 = in.n[0];
          n1 = in.n[1];
          n2 = in.n[2];
          bcbase = in.bc_off + (long long)band * in.ncells;
          coff = in.cell_off;
          vtm = A.vtm32[(long long)inst * A.nb + band];
          all_real = A.all_real[(long long)inst * A.nb + band] != 0;
        }
        const InstDesc& in = A.inst[inst];
        const unsigned local = pid - g_first;
        const int q = (int)udiv(local, (unsigned)g_ne, g_mag);
        int e = (int)(local - (unsigned)q * (unsigned)g_ne);
        if (g_perm >= 0) e = A.perm[g_perm + e];
        if (kind == 0) {
          w = A.coef[bcbase + e];
          if (!ADJ) {
            double Te = A.T[coff + e];
            if (A.srcshift) Te += A.srcshift[coff + e];
            w *= Te;
          }
        } else {
          w = A.wcoef[((long long)inst * A.nb + band) * 6 + kind - 1];
          if (!ADJ) w *= A.wallTf[in.bface_off + in.wface_off[kind - 1] + e];
          if (ADJ && (acc_slot != kind - 1 || acc_inst != inst)) {
            flush_wall();
            acc_slot = kind - 1;
            acc_inst = inst;
          }
        }
        if ((__double_as_longlong(w) << 1) != 0) {
          int c[3];
          uint32_t id;
          float s[3];
          emitter = e;
          emitter_cell<DIM>(in, S, inst, kind, e, c, id);
          st.init(A.seed, in.inst_id, (uint32_t)band, A.epoch, id, (uint32_t)q);
          emit_segment<DIM>(st, kind, xi, s);
#pragma unroll
          for (int a = 0; a < DIM; ++a) {
            g[a] = s[a] * __frcp_rn(in.hf[a]);
            lo[a] = (float)-c[a];
            hi[a] = (float)((a == 0 ? n0 : (a == 1 ? n1 : n2)) - c[a]);
          }
          cell0 = c[0] + n0 * (c[1] + n1 * c[2]);
          ub = all_real ? 0u : st.even_word();
          st.j += 2;
          D = __fmul_rn(-__logf(word_uniform<float>(st.first)), vtm);
          eD = fmaf(D, TIE_LOG_REL, vtm * TIE_LOG_ABS);
          alive = true;
        }
      }
      rbeg += take;
    }
    if (!__any_sync(0xffffffffu, alive)) {
      if (exhausted) break;
      continue;
    }
    if (alive && st.j >= L.max_j) {  // FP64 tracking: the replay keeps the step budget
      land_defer(S, pid);
      alive = false;
    }
    if (alive) {
#pragma unroll 1
      for (int it = 0; it < S.walk_k; ++it) {
        if (it > 0 && __popc(__activemask()) < WALK_MIN_LANES) break;
        const float rel = fmaf(D, LAND_REL, eD);
        bool out = false, in_dom = true, near = false;
        int o[3] = {0, 0, 0};
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
          const float X = fmaf(g[a], D, xi[a]), tol = fmaf(fabsf(g[a]), rel, LAND_ABS);
          out |= lo[a] - X > tol || X - hi[a] > tol;
          in_dom = in_dom && X - lo[a] > tol && hi[a] - X > tol && tol < 0.5f;
          o[a] = floor_near(X, tol, near);
        }
        if (out) {  // absorbed by a wall
          alive = false;
          break;
        }
        // at the first wall within rounding, or a bound beyond the neighbouring cells
        bool real = all_real, defer = !in_dom;
        const int cell = cell0 + o[0] + (DIM >= 2 ? n0 * o[1] : 0) + (DIM == 3 ? n0 * n1 * o[2] : 0);
        if (!defer) {
          if (all_real) {
            defer = near;
          } else {
            // rejected wherever it lies within the bound when the draw exceeds the largest ratio
            // of the cell's neighbourhood; otherwise the cell and the ratio must be certain
            const float ua = word_uniform<float>(ub);
            if (ua - A.ratio_nb32[bcbase + cell] < TIE_ACC) {
              const float ra = A.ratio32[bcbase + cell];
              defer = near || fabsf(ua - ra) < TIE_ACC;
              real = ua < ra;
            }
          }
        }
        if (defer) {
          land_defer(S, pid);
          alive = false;
          break;
        }
        if (real) {
          if (ADJ) {
            const double val = w * L.lamVm[coff + cell];
            if (kind == 0) atomicAdd(&A.adj_out[coff + emitter], val);
            else acc += val;
          } else {
            deposit<K32>(A, S, bcbase + cell, w);
          }
          alive = false;
          break;
        }
        uint32_t uw;
        st.next_pair(uw, ub);
        const float ell = __fmul_rn(-__logf(word_uniform<float>(uw)), vtm);
        D = __fadd_rn(D, ell);
        eD = fmaf(D, TIE_SUM, fmaf(ell, TIE_LOG_REL, eD + vtm * TIE_LOG_ABS));
      }
    }
  }
  if (ADJ) flush_wall();
}

__global__ void lam_over_vm_kernel(long long n, const double* lam, const double* invVm, double* out) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    out[i] = lam[i] * invVm[i];
}

template <int DIM, bool ADJ, bool K32>
cudaError_t launch_dim(const Ctx* c, const SweepArgs& a, const StagedArgs& S, const LandArgs& L, cudaStream_t s) {
  const void* f = c->all_real_all ? (const void*)land_kernel<DIM, ADJ, K32> : (const void*)land_chain_kernel<DIM, ADJ, K32>;
  int nb = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f, LAND_NT, 0);
  if (e != cudaSuccess) return e;
  // warps beyond the work would only claim and leave
  const long long warps = c->all_real_all ? (long long)L.n_tasks : (a.total_particles + S.warp_grab - 1) / S.warp_grab;
  const long long want = (warps * 32 + LAND_NT - 1) / LAND_NT;
  const int blocks = (int)std::max<long long>(1, std::min<long long>(want, (long long)c->sm_count * std::max(nb, 1)));
  if (c->all_real_all) land_kernel<DIM, ADJ, K32><<<blocks, LAND_NT, 0, s>>>(a, S, L);
  else land_chain_kernel<DIM, ADJ, K32><<<blocks, LAND_NT, 0, s>>>(a, S, L);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_land(const Ctx* c, const SweepArgs& a, bool adj, cudaStream_t s) {
  StagedArgs S = {};
  S.warp_grab = c->opt.warp_grab > 0 ? c->opt.warp_grab : 256;
  S.walk_k = c->opt.walk_k > 0 ? c->opt.walk_k : 16;
  S.group_mag = adj ? c->d_all_group_mag : c->d_group_mag;
  S.mag_n0 = c->d_mag;
  S.mag_n1 = c->d_mag + c->n_inst;
  S.mag_wall = c->d_mag + 2 * c->n_inst;
  S.defer = c->d_defer;
  S.defer_n = c->d_defer_n;
  S.defer_cap = c->defer_cap;
  S.over = c->d_over;
  S.over_words = (unsigned)((a.total_particles + 31) / 32);
  S.err = c->d_err;
  const bool k32 = !adj && c->opt.tally == IUGKP_TALLY_STAGED_K32;
  S.R32 = k32 ? c->d_R32 : nullptr;
  LandArgs L;
  L.groups = adj ? c->d_land_all : c->d_land_fwd;
  L.n_groups = a.n_groups;
  L.n_tasks = adj ? c->land_all_tasks : c->land_fwd_tasks;
  L.qch = adj ? c->land_all_qch : c->land_fwd_qch;
  L.next = reinterpret_cast<unsigned long long*>(c->d_defer_n + 2);
  L.lamVm = c->d_work;
  // two uniforms per candidate; FP32 tracking follows a chain to its end, as its full sweep does
  L.max_j = c->opt.precision == IUGKP_TRACK_FP64 ? 2u * EXACT_MAX_CANDIDATES : 0xffffffffu;
  const size_t bc = (size_t)c->nb * c->total_cells;
  PrologueArgs P = {};
  auto clear = [&](void* p, size_t n) {
    P.clear[P.n_clear] = reinterpret_cast<unsigned long long*>(p);
    P.words[P.n_clear++] = (long long)n;
  };
  clear(c->d_defer_n, 2);  // queue length and claim counter
  if (adj) {
    clear(a.adj_out, (size_t)c->total_cells);
    clear(a.adj_wall, (size_t)c->total_walls);
  } else if (k32) {
    clear(c->d_R32, bc);
  } else {
    clear(a.R, bc);
  }
  cudaError_t e = launch_prologue(c, a, P, s);
  if (e != cudaSuccess) return e;
  if (adj) {
    // lambda / (V m), gathered by every particle: into the correction solve's scratch, free
    // until the correction that follows on the same stream
    lam_over_vm_kernel<<<(unsigned)std::min<long long>((c->total_cells + 255) / 256, 8ll * c->sm_count), 256, 0, s>>>(
        c->total_cells, a.lambda, a.invVm, c->d_work);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    switch (c->dim) {
      case 1: e = launch_dim<1, true, false>(c, a, S, L, s); break;
      case 2: e = launch_dim<2, true, false>(c, a, S, L, s); break;
      default: e = launch_dim<3, true, false>(c, a, S, L, s); break;
    }
    if (e != cudaSuccess) return e;
    return launch_adjoint_replay(c, a, S, s);
  }
  if (k32) {
    switch (c->dim) {
      case 1: e = launch_dim<1, false, true>(c, a, S, L, s); break;
      case 2: e = launch_dim<2, false, true>(c, a, S, L, s); break;
      default: e = launch_dim<3, false, true>(c, a, S, L, s); break;
    }
    if (e != cudaSuccess) return e;
    if ((e = launch_k32_finalize(c, c->d_R32, a.R, (long long)bc, s)) != cudaSuccess) return e;
  } else {
    switch (c->dim) {
      case 1: e = launch_dim<1, false, false>(c, a, S, L, s); break;
      case 2: e = launch_dim<2, false, false>(c, a, S, L, s); break;
      default: e = launch_dim<3, false, false>(c, a, S, L, s); break;
    }
    if (e != cudaSuccess) return e;
  }
  return launch_replay(c, a, S, s);  // the deferred particles, in FP64
}

// Tasks of a sweep over a group list: tiles of at most 32 emitters (equal widths;
// narrow groups put several particles of an emitter side by side), qch particles per emitter and
// task: at most qch_max, fewer where that would leave warps without work.
// join: the groups of one instance and kind over its bands form a chain whose passes are numbered
// through (where all of them visit their emitters in emitter order); only a chain's first group
// has tasks then.
void land_tasks(const Ctx* c, const std::vector<Group>& groups, std::vector<LandGroup>& out, unsigned& n_tasks, int& qch,
                int qch_max, int warps_per_sm, bool join) {
  long long total = 0;
  for (const Group& g : groups) total += (long long)g.n_emitters * g.per_emitter;
  const long long warps = (long long)std::max(1, c->sm_count) * warps_per_sm;
  qch = (int)std::max<long long>(1, std::min<long long>(qch_max, total / (32 * 4 * warps)));
  out.clear();
  for (const Group& g : groups) {
    LandGroup l;
    l.first = (unsigned)g.first_particle;
    l.inst = g.inst;
    l.band = g.band;
    l.kind = g.kind;
    l.ne = g.n_emitters;
    l.per = g.per_emitter;
    l.perm_off = g.perm_off;
    l.ntile = (g.n_emitters + 31) / 32;
    l.tw = (g.n_emitters + l.ntile - 1) / l.ntile;
    l.reps = 32 / l.tw;
    l.next = -1;
    l.pass0 = 0;
    out.push_back(l);
  }
  std::vector<long long> passes(out.size());
  std::vector<char> joined(out.size(), 0);
  for (size_t g = 0; g < out.size(); ++g) passes[g] = (out[g].per + out[g].reps - 1) / out[g].reps;
  if (join) {
    for (size_t g0 = 0; g0 < out.size();) {  // one instance at a time
      size_t g1 = g0;
      while (g1 < out.size() && out[g1].inst == out[g0].inst) ++g1;
      std::vector<int> last(7, -1);
      std::vector<size_t> head(7, 0);
      for (size_t g = g0; g < g1; ++g) {
        const int k = out[g].kind;
        if (out[g].perm_off >= 0) continue;
        if (last[k] >= 0) {
          out[last[k]].next = (int)g;
          out[g].pass0 = (int)passes[head[k]];
          passes[head[k]] += passes[g];
          joined[g] = 1;
        } else {
          head[k] = g;
        }
        last[k] = (int)g;
      }
      g0 = g1;
    }
  }
  // a chained group gets no tasks (the search for a task's group takes the last group that starts at
  // or before it: never one whose start is the next head's)
  long long t0 = 0;
  for (size_t g = 0; g < out.size(); ++g) {
    out[g].task0 = (unsigned)t0;
    if (!joined[g]) t0 += (long long)out[g].ntile * ((passes[g] + qch - 1) / qch);
  }
  n_tasks = (unsigned)t0;
}

}  // namespace iugkp
