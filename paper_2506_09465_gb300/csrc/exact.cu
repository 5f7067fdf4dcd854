// Filtered FP64 sweep: the sweep of contexts with FP64 tracking. Every decision of a particle's
// walk (the cell of each candidate, acceptance, the wall it leaves through, the row of every
// face it crosses) is that of the FP64 positions, directions and paths. It is taken in FP32 where
// an error bound shows that both agree (a floating-point filter: Fortune and Van Wyk, "Efficient
// exact arithmetic for computational geometry", 1993) and in FP64 otherwise. Weights and tallies
// are FP64 throughout. Method: arXiv 2506.09465 Sec. 3.1 steps (1)-(3), Sec. 3.2.
//
// What the plain one-thread-per-particle kernel (sweep.cu) spends its time on is GB300's FP64
// pipe, 2 lanes per clock and SM against 128 in FP32: logarithm, sine and cosine, square root
// and divisions of the emission, and three FP64 operations per face crossed. Here a particle
// costs FP32 instructions and its FP64 atomics.
//
//  * Lanes hold emitters (landing.cuh, land.cu): a warp follows 32 particles to their ends.
//  * Faces: along axis a the k-th face is crossed at xi_q + rho_q (k + delta_a) cells along each
//    other axis q (rho_q = g_q / |g_a|, delta_a the distance to the first face in cells); the
//    floor of that is the face's row. A warp deals its particles' faces to its lanes in segments.
//    A row within the bound of a cell edge is queued and found in FP64.
//  * In 1D the faces a particle crosses are one run (a slab of 50 cells has all of its crossings on
//    51 addresses, whose FP64 atomics serialise at the L2): its weight is added to the O(log faces)
//    nodes of a binary tree over the faces whose leaves make up the run, and a face is the sum over
//    its leaf and the nodes above it. Nothing is subtracted, so a face keeps the digits that its own
//    crossings have, deep in a thick film too, and an infinite or NaN weight stays with the faces it
//    crosses (differences at the ends of the runs and prefix sums kept neither).
//  * Candidates and exits within the bound of a face, a wall, a corner or the acceptance ratio
//    leave the particle to the FP64 replay.
//  * What a wall absorbs is the sum of its faces as tallied; the power it emits is added to them
//    afterwards (closing.cu).
//
// Bounds, in units of 2^-23 relative: g 3.5 (landing.cuh); the wall distance W_a / |g_a|: g, one
// rounding of W and the quotient's 2 ulp, 6 in all; rho 9 and rho (k + delta) 10.5. EXIT_REL and
// ITEM_REL are at least twice those.
#include <cuda_runtime.h>

#include <algorithm>

#include "device.cuh"
#include "internal.h"
#include "landing.cuh"
#include "plain.cuh"
#include "replay.cuh"
#include "staged.h"
#include "walk32.cuh"

namespace iugkp {

namespace {

constexpr float EXIT_REL = 0x1p-18f;
constexpr float ITEM_REL = 0x1.6p-19f;
constexpr int EXACT_SEG = 8;  // faces per segment
constexpr int EXACT_NT = 256;

struct ExactArgs {
  uint2* items;          // queued faces: {forward index, axis << 30 | k}
  unsigned* n_items;
  unsigned cap;
  double* node;          // 1D: [copies][2 faces per instance] nodes of the trees over the faces
  long long node_stride;
  int copies;
};

// Adds w to the run of faces [a, b) of a tree over n faces (leaves at n .. 2 n - 1, the node above i
// at i / 2: the bottom-up tree, which needs no power of two).
__device__ __forceinline__ void add_run(double* node, int n, int a, int b, double w) {
  for (unsigned l = (unsigned)(a + n), r = (unsigned)(b + n); l < r; l >>= 1, r >>= 1) {
    if (l & 1u) atomicAdd(&node[l++], w);
    if (r & 1u) atomicAdd(&node[--r], w);
  }
}

// Emitter-major index of the particle with forward index pid (q-major in its group's visiting order).
__device__ __forceinline__ long long emitter_major(const SweepArgs& A, unsigned pid) {
  const Group G = A.groups[find_group(A.groups, A.n_groups, (long long)pid)];
  const unsigned local = pid - (unsigned)G.first_particle;
  const int q = (int)(local / (unsigned)G.n_emitters);
  int e = (int)(local - (unsigned)q * (unsigned)G.n_emitters);
  if (G.perm_off >= 0) e = A.perm[G.perm_off + e];
  return G.first_particle + (long long)e * G.per_emitter + q;
}

// Tallies of a replayed particle: every face as it is crossed; W as w (scaled by tau_maj after the
// sweep, or set to tau_maj R in all-real bands) from candidate k_done on.
struct ReplayTally {
  const SweepArgs& A;
  const InstDesc& in;
  double w;
  int k_done;
  bool all_real;
  __device__ bool candidate(int k, long long ci) {
    if (k < k_done) return false;
    if (A.W && !all_real) atomicAdd(&A.W[ci], w);
    return true;
  }
  __device__ void real(long long ci, int) { atomicAdd(&A.R[ci], w); }
  __device__ void cross(int, int stp, long long face) {
    if (A.F) atomicAdd(&A.F[in.face_off + face], stp > 0 ? w : -w);
  }
  __device__ void exit(int, int, long long) {}
};

template <int DIM>
__device__ void replay_particle(const SweepArgs& A, unsigned pid, int k_done, Counts& cnt) {
  int gi;
  double w;
  Walk<double, DIM> wk;
  Stream st;
  if (!emit_particle<double, DIM, false>(A, emitter_major(A, pid), gi, w, wk, st)) return;
  const Group G = A.groups[gi];
  const InstDesc& in = A.inst[G.inst];
  ReplayTally pol{A, in, w, k_done, A.all_real[(long long)G.inst * A.nb + G.band] != 0};
  walk_particle<double, DIM>(A, in, G.inst, G.band, wk, st, cnt, pol);
}

// The k-th face normal to axis a that a particle crosses, its row found in FP64.
template <int DIM>
__device__ void replay_item(const SweepArgs& A, unsigned pid, int a, int k) {
  int gi;
  double w;
  Walk<double, DIM> wk;
  Stream st;
  if (!emit_particle<double, DIM, false>(A, emitter_major(A, pid), gi, w, wk, st)) return;
  const InstDesc& in = A.inst[A.groups[gi].inst];
  int c[3] = {0, 0, 0};
  double T = 0.0;
#pragma unroll
  for (int o = 0; o < DIM; ++o)
    if (o == a) T = wk.tmax[o] + (double)k * wk.tdelta[o];
  int stp = 1;
#pragma unroll
  for (int o = 0; o < DIM; ++o) {
    if (o == a) {
      stp = wk.step[o];
      c[o] = stp > 0 ? wk.idx[o] + 1 + k : wk.idx[o] - k;
    } else {
      const double d = wk.tdelta[o];
      const int n = count_before64(T, wk.tmax[o], d < RealTraits<double>::inf() ? 1.0 / d : 0.0);
      const int m = wk.step[o] > 0 ? in.n[o] - wk.idx[o] : wk.idx[o] + 1;
      c[o] = wk.idx[o] + wk.step[o] * min(n, m - 1);
    }
  }
  const long long m0 = in.n[0] + (a == 0), m1 = in.n[1] + (a == 1);
  atomicAdd(&A.F[in.face_off + in.fax_off[a] + c[0] + m0 * (c[1] + m1 * c[2])], stp > 0 ? w : -w);
}

// Full queues: done at once by the lane that found the case.
template <int DIM>
__device__ __noinline__ void replay_now(const SweepArgs& A, unsigned pid, int k_done) {
  Counts cnt;
#pragma unroll
  for (int k = 0; k < CNT_N; ++k) cnt.v[k] = 0;
  replay_particle<DIM>(A, pid, k_done, cnt);
#pragma unroll
  for (int k = 0; k < CNT_N; ++k)
    if (cnt.v[k]) atomicAdd(&A.counters[k], cnt.v[k]);
}
template <int DIM>
__device__ __noinline__ void item_now(const SweepArgs& A, unsigned pid, int a, int k) { replay_item<DIM>(A, pid, a, k); }

// A lane's list of faces along one axis, as the warp's lanes read it.
struct ItemList {
  unsigned base;   // face at k = 0, in the emission cell's row
  int step;        // face index step per k
  float xi1, rho1, xi2, rho2, delta;
  unsigned pid;
  double w;        // signed along the axis
  int n, first;    // faces; first segment
};

// The warp tallies its lanes' lists along axis a together: cut into segments of EXACT_SEG faces,
// numbered in lane order and dealt round-robin.
template <int DIM>
__device__ __forceinline__ void tally_lists(const SweepArgs& A, const ExactArgs& X, ItemList* tab, ItemList l, int a,
                                            double* F, int st1, int st2) {
  const int lane = threadIdx.x & 31;
  const int nseg = (l.n + EXACT_SEG - 1) / EXACT_SEG;
  int incl = nseg;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  if (total == 0) return;
  const int first = incl - nseg;
  const unsigned nonempty = __ballot_sync(0xffffffffu, nseg > 0);
  if (nseg > 0) {
    l.first = first;
    tab[__popc(nonempty & ((1u << lane) - 1u))] = l;
  }
  __syncwarp();
  for (int r0 = 0; r0 < total; r0 += 32) {
    const bool starts_here = nseg > 0 && first >= r0 && first < r0 + 32;
    const unsigned bits = __reduce_or_sync(0xffffffffu, starts_here ? 1u << (first - r0) : 0u);
    const int before = __popc(__ballot_sync(0xffffffffu, nseg > 0 && first < r0));
    const int s = r0 + lane;
    if (s >= total) continue;
    const ItemList m = tab[before + __popc(bits & (0xffffffffu >> (31 - lane))) - 1];
    const int k0 = (s - m.first) * EXACT_SEG, k1 = min(m.n, k0 + EXACT_SEG);
    float pos = small_int_float(k0) + m.delta;
    for (int k = k0; k < k1; ++k, pos += 1.f) {
      bool near = false;
      unsigned face = m.base + (unsigned)(k * m.step);
      if (DIM >= 2) {
        const float d1 = m.rho1 * pos;
        face += (unsigned)(st1 * floor_near(m.xi1 + d1, fmaf(fabsf(d1), ITEM_REL, LAND_ABS), near));
      }
      if (DIM == 3) {
        const float d2 = m.rho2 * pos;
        face += (unsigned)(st2 * floor_near(m.xi2 + d2, fmaf(fabsf(d2), ITEM_REL, LAND_ABS), near));
      }
      if (!near) {
        atomicAdd(&F[face], m.w);
      } else {
        const unsigned j = atomicAdd(X.n_items, 1u);
        if (j < X.cap) X.items[j] = make_uint2(m.pid, ((unsigned)a << 30) | (unsigned)k);
        else item_now<DIM>(A, m.pid, a, k);
      }
    }
  }
  __syncwarp();
}

template <int DIM>
__global__ void __launch_bounds__(EXACT_NT) exact_kernel(SweepArgs A, StagedArgs S, LandArgs L, ExactArgs X) {
  __shared__ ItemList s_tab[DIM == 1 ? 1 : EXACT_NT / 32][DIM == 1 ? 1 : 32];
  const int lane = threadIdx.x & 31;
  ItemList* tab = s_tab[DIM == 1 ? 0 : threadIdx.x >> 5];
  unsigned n_fl = 0, n_cand = 0, n_real = 0, n_cross = 0, n_exit = 0;
  TaskGroup tg;
  for (;;) {
    unsigned task = 0;
    if (lane == 0) task = (unsigned)atomicAdd(L.next, 1ull);
    task = __shfl_sync(0xffffffffu, task, 0);
    if (task >= L.n_tasks) break;
    tg.find(L, task);
    const LandGroup& G = L.groups[tg.gi];
    const unsigned t = task - tg.t_beg;
    const int qc = (int)(t / (unsigned)G.ntile), tile = (int)(t - (unsigned)qc * (unsigned)G.ntile);
    const InstDesc& in = A.inst[G.inst];
    LaneEmitter<DIM> em;
    em.template init<false>(A, S, G, in, tile, lane);
    const int n0 = in.n[0], n1 = in.n[1], n2 = in.n[2], kb = G.inst * A.nb + G.band;
    const float vtm = A.vtm32[kb], va = vtm * TIE_LOG_ABS;
    const bool all_real = A.all_real[kb] != 0;
    const long long bcbase = in.bc_off + (long long)G.band * in.ncells;
    const uint32_t inst_id = in.inst_id;
    double* F = A.F ? A.F + in.face_off : nullptr;
    double* node = DIM == 1 && A.F ? X.node + (blockIdx.x % (unsigned)X.copies) * X.node_stride + 2 * in.face_off : nullptr;
    const int qbeg = qc * (L.qch * G.reps) + em.sub, qend = min(G.per, (qc + 1) * (L.qch * G.reps));
    for (int j = 0; j < L.qch; ++j) {
      const int q = qbeg + j * G.reps;
      const bool act = em.on && q < qend;
      if (!__any_sync(0xffffffffu, act)) break;
      int items[3] = {0, 0, 0};
      float xi[3] = {0.f, 0.f, 0.f}, g[3] = {0.f, 0.f, 0.f};
      const unsigned pid = G.first + (unsigned)q * (unsigned)G.ne + (unsigned)em.rank;
      if (act) {
        n_fl += 1;
        Stream st;
        st.init(A.seed, inst_id, (uint32_t)G.band, A.epoch, em.id, (uint32_t)q);
        {
          float s[3];
          emit_segment<DIM>(st, G.kind, xi, s);
#pragma unroll
          for (int a = 0; a < DIM; ++a) g[a] = s[a] * em.ih[a];
        }
        uint32_t ub = all_real ? 0u : st.even_word();
        st.j += 2;
        float D = __fmul_rn(-__logf(word_uniform<float>(st.first)), vtm);
        float eD = fmaf(D, TIE_LOG_REL, va);
        bool out = false, defer = false;
        int o[3] = {0, 0, 0}, kc = 0;
#pragma unroll 1
        for (;;) {
          const float rel = fmaf(D, LAND_REL, eD);
#pragma unroll
          for (int a = 0; a < DIM; ++a) {
            const float P = fmaf(g[a], D, xi[a]), tol = fmaf(fabsf(g[a]), rel, LAND_ABS);
            out |= em.lo[a] - P > tol || P - em.hi[a] > tol;  // beyond a wall for the FP64 walk too
            o[a] = floor_near(P, tol, defer);
          }
          if (out) {
            defer = false;
            break;
          }
          if (defer) break;
          const int cell = em.cell0 + o[0] + (DIM >= 2 ? n0 * o[1] : 0) + (DIM == 3 ? n0 * n1 * o[2] : 0);
          const long long ci = bcbase + cell;
          bool real = all_real;
          if (!all_real) {
            const float ua = word_uniform<float>(ub), ra = A.ratio32[ci];
            if (fabsf(ua - ra) < TIE_ACC) {
              defer = true;
              break;
            }
            real = ua < ra;
            if (A.W) atomicAdd(&A.W[ci], em.w);
          }
          ++kc;
          if (real) {
            n_real += 1;
            atomicAdd(&A.R[ci], em.w);
            break;
          }
          if (kc >= EXACT_MAX_CANDIDATES) {  // the replay keeps the step budget
            defer = true;
            break;
          }
          uint32_t uw;
          st.next_pair(uw, ub);
          const float ell = __fmul_rn(-__logf(word_uniform<float>(uw)), vtm);
          D = __fadd_rn(D, ell);
          eD = fmaf(D, TIE_SUM, fmaf(ell, TIE_LOG_REL, eD + va));
        }
        n_cand += kc;
        int p = -1;  // the axis of the wall it leaves through
        if (out) {
          float te = INFINITY, te2 = INFINITY;  // wall distances: the nearest and the next
#pragma unroll
          for (int a = 0; a < DIM; ++a) {
            const float ta = __fdividef(g[a] > 0.f ? em.hi[a] - xi[a] : xi[a] - em.lo[a], fabsf(g[a]));
            if (ta < te) {
              te2 = te;
              te = ta;
              p = a;
            } else {
              te2 = fminf(te2, ta);
            }
          }
          defer = DIM > 1 && te2 - te <= EXIT_REL * te;
#pragma unroll
          for (int a = 0; a < DIM; ++a) {
            const float dx = g[a] * te;
            if (a != p) o[a] = floor_near(xi[a] + dx, fmaf(fabsf(dx), EXIT_REL, LAND_ABS), defer);
          }
        }
        if (defer) {
          const unsigned i = atomicAdd(S.defer_n, 1u);
          if (i < S.defer_cap) S.defer[i] = make_uint2(pid, (unsigned)kc);
          else replay_now<DIM>(A, pid, kc);
        } else {
          n_exit += out ? 1 : 0;
#pragma unroll
          for (int a = 0; a < DIM; ++a) {
            // interior faces crossed; on the exit axis all of them, and the wall's face
            const int c = a == p ? (g[a] > 0.f ? (a == 0 ? n0 : (a == 1 ? n1 : n2)) - 1 - em.c[a] : em.c[a]) : abs(o[a]);
            n_cross += c;
            items[a] = c + (a == p ? 1 : 0);
          }
          if (DIM == 1 && node && items[0] > 0) {
            if (g[0] > 0.f) add_run(node, n0 + 1, em.c[0] + 1, em.c[0] + 1 + items[0], em.w);
            else add_run(node, n0 + 1, em.c[0] + 1 - items[0], em.c[0] + 1, -em.w);
          }
        }
      }
      if (DIM > 1 && F) {
#pragma unroll
        for (int a = 0; a < DIM; ++a) {
          // the other axes in index order, and the face index steps along them
          const int q1 = a == 0 ? 1 : 0, q2 = a == 2 ? 1 : 2;
          const int m0 = n0 + (a == 0), m1 = n1 + (a == 1);
          const int stride[3] = {1, m0, m0 * m1};
          const float ig = __fdividef(1.f, fabsf(g[a]));
          ItemList l;
          l.base = (unsigned)in.fax_off[a] + (unsigned)(em.c[0] + m0 * (em.c[1] + m1 * em.c[2])) +
                   (g[a] > 0.f ? (unsigned)stride[a] : 0u);
          l.step = g[a] > 0.f ? stride[a] : -stride[a];
          l.xi1 = xi[q1];
          l.rho1 = g[q1] * ig;
          l.xi2 = DIM == 3 ? xi[q2] : 0.f;
          l.rho2 = DIM == 3 ? g[q2] * ig : 0.f;
          l.delta = g[a] > 0.f ? 1.f - xi[a] : xi[a];
          l.pid = pid;
          l.w = g[a] > 0.f ? em.w : -em.w;
          l.n = items[a];
          l.first = 0;
          tally_lists<DIM>(A, X, tab, l, a, F, stride[q1], stride[q2]);
        }
      }
    }
  }
  unsigned long long v[5] = {n_fl, n_cand, n_real, n_cross, n_exit};
  const int slot[5] = {CNT_FLIGHTS, CNT_CANDIDATES, CNT_REAL, CNT_CROSSINGS, CNT_WALL_EXITS};
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    unsigned long long x = v[i];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) x += __shfl_down_sync(0xffffffffu, x, d);
    if (lane == 0 && x) atomicAdd(&A.counters[slot[i]], x);
  }
}

// The queued particles, then the queued faces, one thread each.
template <int DIM>
__global__ void __launch_bounds__(64) exact_replay_kernel(SweepArgs A, StagedArgs S, ExactArgs X) {
  Counts cnt;
#pragma unroll
  for (int k = 0; k < CNT_N; ++k) cnt.v[k] = 0;
  // warp j of every block numbered before warp j + 1 of any: a short queue is spread over the SMs
  const unsigned wid = (threadIdx.x >> 5) * gridDim.x + blockIdx.x, lane = threadIdx.x & 31;
  const unsigned step = gridDim.x * blockDim.x;
  const unsigned n = min(*S.defer_n, S.defer_cap), ni = min(*X.n_items, X.cap);
  for (unsigned i = 32u * wid + lane; i < n; i += step) replay_particle<DIM>(A, S.defer[i].x, (int)S.defer[i].y, cnt);
  if (DIM > 1)
    for (unsigned i = 32u * wid + lane; i < ni; i += step) {
      const uint2 it = X.items[i];
      replay_item<DIM>(A, it.x, (int)(it.y >> 30), (int)(it.y & 0x3fffffffu));
    }
#pragma unroll
  for (int k = 0; k < CNT_N; ++k) {
    unsigned long long x = cnt.v[k];
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) x += __shfl_down_sync(0xffffffffu, x, d);
    if (lane == 0 && x) atomicAdd(&A.counters[k], x);
  }
}

template <int DIM>
cudaError_t launch_dim(const Ctx* c, const SweepArgs& a, const StagedArgs& S, const LandArgs& L, const ExactArgs& X,
                       cudaStream_t s) {
  int nb = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, exact_kernel<DIM>, EXACT_NT, 0);
  if (e != cudaSuccess) return e;
  const long long want = ((long long)L.n_tasks * 32 + EXACT_NT - 1) / EXACT_NT;
  const int blocks = (int)std::max<long long>(1, std::min<long long>(want, (long long)c->sm_count * std::max(nb, 1)));
  exact_kernel<DIM><<<blocks, EXACT_NT, 0, s>>>(a, S, L, X);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  exact_replay_kernel<DIM><<<c->sm_count * 8, 64, 0, s>>>(a, S, X);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_exact(const Ctx* c, const SweepArgs& a, cudaStream_t s) {
  StagedArgs S = {};
  S.group_mag = c->d_group_mag;
  S.mag_n0 = c->d_mag;
  S.mag_n1 = c->d_mag + c->n_inst;
  S.mag_wall = c->d_mag + 2 * c->n_inst;
  S.defer = c->d_defer;
  S.defer_n = c->d_defer_n;
  S.defer_cap = c->defer_cap;
  S.err = c->d_err;
  LandArgs L = {};
  L.groups = c->d_sync_groups;
  L.n_groups = a.n_groups;
  L.n_tasks = c->sync_tasks;
  L.qch = c->sync_qch;
  L.next = reinterpret_cast<unsigned long long*>(c->d_defer_n + 2);
  ExactArgs X = {};
  X.items = c->d_items;
  X.n_items = c->d_defer_n + 1;
  X.cap = c->items_cap;
  X.node = c->d_nodes;
  X.node_stride = 2 * c->total_faces;
  X.copies = c->node_copies;
  PrologueArgs P = {};
  auto clear = [&](void* p, size_t n) {
    if (!p || !n) return;
    P.clear[P.n_clear] = reinterpret_cast<unsigned long long*>(p);
    P.words[P.n_clear++] = (long long)n;
  };
  clear(a.R, (size_t)c->nb * c->total_cells);
  if (!c->all_real_all) clear(a.W, (size_t)c->nb * c->total_cells);  // else W = tau_maj R afterwards
  clear(a.F, (size_t)c->total_faces);
  clear(a.counters, CNT_N);
  clear(c->d_defer_n, 2);
  if (c->dim == 1 && a.F) clear(c->d_nodes, (size_t)X.copies * X.node_stride);
  cudaError_t e = launch_prologue(c, a, P, s);
  if (e != cudaSuccess) return e;
  switch (c->dim) {
    case 1: e = launch_dim<1>(c, a, S, L, X, s); break;
    case 2: e = launch_dim<2>(c, a, S, L, X, s); break;
    default: e = launch_dim<3>(c, a, S, L, X, s); break;
  }
  if (e != cudaSuccess) return e;
  // W scaled, the walls' absorbed power, the walls' emission added to their faces
  return launch_close_tallied(c, a, s);
}

}  // namespace iugkp
