// Inexact-Newton correction solver (arXiv 2506.09465 Sec. 3.3, Eq. "linear-q"): CG on the
// finite-volume diffusion operator, FP64 iterates and residual, preconditioned by one
// aggregation-multigrid V-cycle in FP32; separable operators by fast diagonalization.
//
// One team of thread blocks per instance, one block per SM. Small instances: a team is one thread-block
// cluster (ClusterTeam). Larger or many ones: all blocks resident together (a cooperative launch: it
// starts once a block fits on each SM it needs), the SMs dealt to the instances by their cost
// (plan_teams). A team's blocks split each level's cells in contiguous ranges, exchange neighbour
// values through global memory (L2) between team barriers, and reduce dot products in a fixed rank
// order (every block gets the same value, so all take the same branch). With one 8-block cluster per instance
// the largest of four boxes (64^3, 64 cells per thread and phase) set the time on 8 of 152 SMs:
// 5.5 ms per solve of 11 CG steps, now 1.4 ms (latency of L2 round trips and of the barriers, one
// instruction in six cycles issued; the loads of two cells in flight at once cost 8 % in index
// arithmetic).
// The V-cycle: damped Jacobi smoothing (two sweeps before and two after), restriction by summing
// the children (P^T), Galerkin coarse operators P^T A P built on the host, prolongation by
// injection scaled by alpha (the usual over-correction of piecewise-constant
// aggregation), dense inverse on the coarsest level. It is symmetric, so CG stays CG.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "internal.h"
#include "mg.h"

namespace iugkp {

constexpr int MG32_PASSES_FD = 6;  // refinement passes of the fast diagonalization solve at most
constexpr int MG_NT = 1024;        // threads per block, multigrid CG
constexpr int MG_SMALL_NT = 512;   // ... where every instance is small: fewer warps per barrier
constexpr int MG_CLUSTER = 8;      // blocks of a cluster team
constexpr int FD_NT = 512;         // ... fast diagonalization
// Polls of a team barrier (an L2 round trip each) before a block gives up: a second or so.
constexpr unsigned TEAM_SPIN_LIMIT = 1u << 21;

// The team a block belongs to and the instances the team solves, one after the other.
struct TeamDesc {
  int first_block, size;
  int inst_beg, inst_end;  // into the plan's instance order
};

// The right-hand side and what becomes of the solution x. Newton step: rhs = (sum_b R_b - T V m) / V,
// out = half + theta x (theta per instance). Adjoint: half = at + g, rhs = half - lam,
// out = half + theta_m x (per cell).
struct CorrectionIO {
  const double* R;
  const double* T;
  const double* Vm;
  const double* theta;
  const double* at;        // null: Newton step
  const double* g;
  const double* lam;
  const double* theta_m;
  const double* half;      // Newton: T_half
  double* half_out;        // adjoint: at + g
  double* out;
};

struct MGArgs {
  const InstMG* mg;         // [n_inst]
  const InstDesc* inst;     // [n_inst]
  int nb;
  const TeamDesc* teams;    // of this kernel's plan
  const int* block_team;    // [blocks] team of each block
  const int* order;         // instances, team by team
  unsigned* bar;            // [2 * teams] barrier arrivals, blocks that have left (0 between launches)
  double* slots;            // [blocks * 4] partial sums of the blocks
  int* err;
  CorrectionIO io;
  const double* diag;       // fine FP64 operator
  const double* cx;
  const double* cy;
  const double* cz;
  const float* ldiag;       // all levels, FP32
  const float* ldiag_inv;
  const float* lcx;
  const float* lcy;
  const float* lcz;
  const float* cinv;        // coarsest dense inverses
  const float* fq;          // fast diagonalization: eigenvector matrices
  const float* flam;        // ... and eigenvalues
  float* lb;                // level right-hand sides
  float* lx;                // level iterates
  float* lt;                // level scratch (ping-pong)
  double* rhs;              // [cells]
  double* X;                // [cells] solution
  double* Rr;               // residual
  double* P;
  double* Q;
  double* Z;
  double rtol;
  int maxit;
  int* iters_out;           // [n_inst]
  float alpha, omega;
};

// A block's view of its team.
struct Team {
  int rank, size;
  unsigned* ctr;
  unsigned target;   // arrivals after which the next barrier opens
  int* err;
  double* slots;     // of the team's first block: [2][size][2]
  int buf;
  bool dead;         // a barrier was given up (the same for all threads of the block)
  static constexpr bool solo = false;
  static constexpr long long solo_cells = 4096;  // levels up to here are the first block's alone
  __device__ static float ld(const float* p) { return __ldcg(p); }
  __device__ __forceinline__ int stride() const { return (int)blockDim.x; }
  // What the team's blocks wrote before it is visible to all of them after it.
  __device__ __forceinline__ void sync() {
    __shared__ int s_open;
    if (size == 1) {
      __syncthreads();
      return;
    }
    __syncthreads();
    if (dead) return;
    target += (unsigned)size;
    if (threadIdx.x == 0) {
      // release: what the block's threads wrote before the block barrier; acquire: what the others did
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ctr) : "memory");
      unsigned seen, polls = 0;
      do {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(ctr) : "memory");
      } while ((int)(seen - target) < 0 && ++polls < TEAM_SPIN_LIMIT);
      s_open = (int)(seen - target) >= 0;
      if (!s_open) atomicOr(err, ERR_WAIT);
    }
    __syncthreads();
    dead = !s_open;
  }
  __device__ __forceinline__ void range(int nc, int& lo, int& hi) const {
    const int chunk = (nc + size - 1) / size;
    lo = min(nc, rank * chunk);
    hi = min(nc, lo + chunk);
  }
  // Sums NV values over the whole team in a fixed order; also a barrier.
  template <int NV>
  __device__ __forceinline__ void sum(double (&v)[NV], double* sh) {
    static_assert(NV <= 2, "two values at most");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      double x = v[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
      if (lane == 0) sh[k * 32 + warp] = x;
    }
    __syncthreads();
    double* mine = slots + (size_t)buf * size * 2;
    if (warp < NV) {
      double x = lane < (int)(blockDim.x >> 5) ? sh[warp * 32 + lane] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
      if (lane == 0) mine[rank * 2 + warp] = x;
    }
    sync();
    if (warp < NV) {
      double x = 0.0;
      for (int r = lane; r < size; r += 32) x += __ldcg(&mine[r * 2 + warp]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
      if (lane == 0) sh[64 + warp] = x;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = sh[64 + k];
    buf ^= 1;  // a slot is written again only after the next sum's barrier
  }
};

// The same for a team that is one thread-block cluster (MG_CLUSTER blocks, started together by the
// hardware, so the launch needs nothing else of the device): the cluster's own barrier, which costs a
// third of a round trip through L2, and partial sums read from the blocks' shared memory.
struct ClusterTeam {
  int rank, size;
  double* slots;  // this block's shared memory: [2][2]
  int buf;
  static constexpr bool dead = false, solo = false;
  static constexpr long long solo_cells = 1024;
  __device__ static float ld(const float* p) { return __ldcg(p); }
  __device__ __forceinline__ int stride() const { return (int)blockDim.x; }
  __device__ __forceinline__ void sync() { cooperative_groups::this_cluster().sync(); }
  __device__ __forceinline__ void range(int nc, int& lo, int& hi) const {
    const int chunk = (nc + size - 1) / size;
    lo = min(nc, rank * chunk);
    hi = min(nc, lo + chunk);
  }
  template <int NV>
  __device__ __forceinline__ void sum(double (&v)[NV], double* sh) {
    static_assert(NV <= 2, "two values at most");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      double x = v[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
      if (lane == 0) sh[k * 32 + warp] = x;
    }
    __syncthreads();
    if (warp < NV) {
      double x = lane < (int)(blockDim.x >> 5) ? sh[warp * 32 + lane] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
      if (lane == 0) slots[buf * 2 + warp] = x;
    }
    sync();
    if (warp < NV) {
      double x = lane < size ? *cooperative_groups::this_cluster().map_shared_rank(slots + buf * 2 + warp, lane) : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
      if (lane == 0) sh[64 + warp] = x;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = sh[64 + k];
    buf ^= 1;  // a slot is written again only after the next sum's barrier
  }
};

// The finest level's cells and the order of its FP32 sums. The cells are cut into MG_RANKS equal
// ranges; unit (r, w) has the cells of range r whose offset modulo 32 MG_WARPS falls on 32 w .. 32 w
// + 31, one per lane, in steps: a lane's products are added in FP32 over the steps, the lanes' sums
// in FP64. A team's blocks take whole units, so that the FP32 part of a sum does not depend on how
// many blocks share the instance (the order of the FP64 part does: last bits of the dot products).
// The products are formed in parallel over units and steps and pass through shared
// memory to the warp that adds a unit's.
constexpr int MG_RANKS = 8, MG_WARPS = 16;
constexpr int MG_STAGE = 128;  // unit steps staged at a time

__host__ __device__ __forceinline__ int range_units_log(long long chunk) {
  int l = 0;
  while ((32 << l) < chunk && (1 << l) < MG_WARPS) ++l;
  return l;
}

struct Units {
  int n, chunk, steps, lw;  // cells, cells of a range, steps of a unit, 2^lw units of a range (all that have cells)
  int u0, u1;               // this block's units
  template <class TM>
  __device__ __forceinline__ Units(int cells, const TM& tm) {
    n = cells;
    chunk = (cells + MG_RANKS - 1) / MG_RANKS;
    steps = (chunk + 32 * MG_WARPS - 1) / (32 * MG_WARPS);
    lw = range_units_log(chunk);
    const int all = MG_RANKS << lw, per = (all + tm.size - 1) / tm.size;
    u0 = min(all, tm.rank * per);
    u1 = min(all, u0 + per);
  }
  // Cell of a lane at a unit's step, or -1.
  __device__ __forceinline__ int cell(int unit, int step) const {
    const int r = unit >> lw, o = (unit - (r << lw)) * 32 + (threadIdx.x & 31) + step * (32 * MG_WARPS);
    const int i = r * chunk + o;
    return o < chunk && i < n ? i : -1;
  }
  template <class F>
  __device__ __forceinline__ void each(F f) const {
    const int total = (u1 - u0) * steps;
    for (int e = threadIdx.x >> 5; e < total; e += (int)(blockDim.x >> 5)) {
      const int q = e / steps, i = cell(u0 + q, e - q * steps);
      if (i >= 0) f(i);
    }
  }
  // f(i) returns the NS factors of cell i; out[v] is this thread's share of the sums over the
  // cells of factor A_v x factor B_v (A, B: 4 bits per v).
  template <int NS, int NV, unsigned A, unsigned B, class F>
  __device__ __forceinline__ void dot(F f, float (*stage)[NS * 32], double (&out)[NV]) const {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sg = min(steps, MG_STAGE), ug = MG_STAGE / sg;  // steps, units staged at a time (steps over MG_STAGE: one)
#pragma unroll
    for (int v = 0; v < NV; ++v) out[v] = 0.0;
    float acc[NV];
    for (int ub = u0; ub < u1; ub += ug) {
      const int nu = min(ug, u1 - ub);
      for (int sb = 0; sb < steps; sb += sg) {
        const int ns = min(sg, steps - sb), total = nu * ns;
        for (int e = warp; e < total; e += (int)(blockDim.x >> 5)) {
          const int q = e / ns, i = cell(ub + q, sb + e - q * ns);
          float x[NS];
#pragma unroll
          for (int t = 0; t < NS; ++t) x[t] = 0.f;
          if (i >= 0) f(i, x);
#pragma unroll
          for (int t = 0; t < NS; ++t) stage[e][t * 32 + lane] = x[t];
        }
        __syncthreads();
        for (int u = warp; u < nu; u += (int)(blockDim.x >> 5)) {
          if (sb == 0) {
#pragma unroll
            for (int v = 0; v < NV; ++v) acc[v] = 0.f;
          }
#pragma unroll 4
          for (int st = 0; st < ns; ++st) {
            const float* x = stage[u * ns + st];
#pragma unroll
            for (int v = 0; v < NV; ++v)
              acc[v] = fmaf(x[((A >> (4 * v)) & 15u) * 32 + lane], x[((B >> (4 * v)) & 15u) * 32 + lane], acc[v]);
          }
          if (sb + ns == steps) {
#pragma unroll
            for (int v = 0; v < NV; ++v) out[v] += (double)acc[v];
          }
        }
        __syncthreads();
      }
    }
  }
};

// Levels of at most TM::solo_cells cells go to the team's first block, their vectors in its shared
// memory: the work is small and every phase waits for the previous one, so the barriers and
// L2 round trips are what they would cost on the team.
struct SoloTeam {
  int nt;  // threads: as many as the level has cells, whole warps (a barrier of 32 warps costs more than one of a few)
  static constexpr bool solo = true;
  __device__ static float ld(const float* p) { return *p; }
  __device__ __forceinline__ int stride() const { return nt; }
  __device__ __forceinline__ void sync() const { asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory"); }
  __device__ __forceinline__ void range(int nc, int& lo, int& hi) const {
    lo = 0;
    hi = nc;
  }
};

constexpr long long MG_SMALL_CELLS = 1024;  // instances up to here take one block of a team launch
// Contexts whose largest instance lies in this range take one cluster per instance, as long as all
// clusters run at once. Teams of four to eight blocks spend their time in L2 barriers there, or leave the
// finest level to one block. us per solve (rtol 1e-3), teams / one cluster each: a 400-cell film
// 313 / 290, 1000 cells 683 / 574, 4000 cells 1854 / 1276; a 64 x 64 square 400 / 265, 120 x 120 569 /
// 474; a 16^3 box 316 / 212, 26^3 497 / 462. Outside it: 120 cells (one block) 188 / 191, 160 x 160 at
// rtol 1e-8 1150 / 1199, 32^3 485 / 523.
constexpr long long MG_CLUSTER_FROM = 256, MG_CLUSTER_CELLS = 18000;

// out[i] = f(i) for every cell of a level that falls on this block: the finest level by units (its
// vectors are the CG's), the others in contiguous ranges.
template <class TM, class F>
__device__ __forceinline__ void level_each(const TM& tm, int l, int nc, float* out, F f) {
  if constexpr (!TM::solo) {
    if (l == 0) {
      Units(nc, tm).each([&](int i) { out[i] = f(i); });
      return;
    }
  }
  int lo, hi;
  tm.range(nc, lo, hi);
  for (int i = lo + threadIdx.x; i < hi; i += tm.stride()) out[i] = f(i);
}

__device__ __forceinline__ void level_coords(const int* n, int i, int& x, int& y, int& z) {
  const int t = i / n[0];
  x = i - t * n[0];
  z = t / n[1];
  y = t - z * n[1];
}

// A_l x on level l (FP32 stencil) for one cell; f(j) is the iterate at cell j.
template <class F>
__device__ __forceinline__ float level_apply(const float* dg, const float* cx, const float* cy, const float* cz, F f,
                                             const int* n, int dim, int i, int nc) {
  const int sy = n[0], sz = n[0] * n[1];
  float q = dg[i] * f(i);
  if (i + 1 < nc) q -= cx[i] * f(i + 1);
  if (i >= 1) q -= cx[i - 1] * f(i - 1);
  if (dim >= 2) {
    if (i + sy < nc) q -= cy[i] * f(i + sy);
    if (i >= sy) q -= cy[i - sy] * f(i - sy);
  }
  if (dim >= 3) {
    if (i + sz < nc) q -= cz[i] * f(i + sz);
    if (i >= sz) q -= cz[i - sz] * f(i - sz);
  }
  return q;
}

// A_l u for u = x + alpha P xc (x prolonged from the coarser level's correction xc, P
// injection), for one cell at coordinates (X, Y, Z), without storing u. Neighbours across a
// boundary are skipped by coordinates (their coefficient is zero).
template <class LD>
__device__ __forceinline__ float level_apply_prolonged(const float* dg, const float* cx, const float* cy,
                                                       const float* cz, const float* x, const float* xc, float alpha,
                                                       const int* n, const int* nC, int dim, int i, int X, int Y,
                                                       int Z) {
  auto u = [&](int j, int x0, int y0, int z0) {
    const int J = (x0 >> 1) + nC[0] * ((y0 >> 1) + nC[1] * (z0 >> 1));
    return fmaf(alpha, LD::ld(&xc[J]), LD::ld(&x[j]));
  };
  const int sy = n[0], sz = n[0] * n[1];
  float q = dg[i] * u(i, X, Y, Z);
  if (X + 1 < n[0]) q -= cx[i] * u(i + 1, X + 1, Y, Z);
  if (X >= 1) q -= cx[i - 1] * u(i - 1, X - 1, Y, Z);
  if (dim >= 2) {
    if (Y + 1 < n[1]) q -= cy[i] * u(i + sy, X, Y + 1, Z);
    if (Y >= 1) q -= cy[i - sy] * u(i - sy, X, Y - 1, Z);
  }
  if (dim >= 3) {
    if (Z + 1 < n[2]) q -= cz[i] * u(i + sz, X, Y, Z + 1);
    if (Z >= 1) q -= cz[i - sz] * u(i - sz, X, Y, Z - 1);
  }
  return q;
}

// The vectors of one level (right-hand side b, iterate x, scratch t) and its operator.
struct LevelView {
  const float *dg, *dinv, *cx, *cy, *cz;
  float *b, *x, *t;
};

__device__ __forceinline__ LevelView global_view(const MGArgs& A, const InstMG& m, int l) {
  const long long o = m.off[l];
  return {A.ldiag + o, A.ldiag_inv + o, A.lcx + o, A.lcy + o, A.lcz + o, A.lb + o, A.lx + o, A.lt + o};
}

// Shared-memory layout of the first block's levels ls .. L-1: per level b, x, t of nc floats.
__device__ __forceinline__ LevelView solo_view(const MGArgs& A, const InstMG& m, int l, int ls, float* smem) {
  const long long o = m.off[l];
  long long so = 0;
  for (int j = ls; j < l; ++j) so += 3 * m.nc[j];
  float* base = smem + so;
  const long long nc = m.nc[l];
  return {A.ldiag + o, A.ldiag_inv + o, A.lcx + o, A.lcy + o, A.lcz + o, base, base + nc, base + 2 * nc};
}

// Downward half of the V-cycle on level l: two sweeps from x = 0 into v.x (the first,
// omega D^{-1} b, is formed where the second reads it: one barrier less), and the restriction of
// the residual into vc.b, the right-hand side of level l + 1 (each child's residual formed where
// it is summed).
template <class TM>
__device__ void vdown(const MGArgs& A, const InstMG& m, int l, const LevelView& v, const LevelView& vc, TM& tm) {
  const int nc = (int)m.nc[l], dim = m.dim;
  const int n[3] = {m.n[l][0], m.n[l][1], m.n[l][2]};
  const float omega = A.omega;
  auto first = [&](int j) { return __fmul_rn(__fmul_rn(omega, TM::ld(&v.b[j])), v.dinv[j]); };
  level_each(tm, l, nc, v.x, [&](int i) {
    const float ax = level_apply(v.dg, v.cx, v.cy, v.cz, first, n, dim, i, nc);
    return first(i) + omega * (TM::ld(&v.b[i]) - ax) * v.dinv[i];
  });
  tm.sync();
  const int ncc = (int)m.nc[l + 1];
  const int* nC = m.n[l + 1];
  int clo, chi;
  tm.range(ncc, clo, chi);
  auto at = [&](int j) { return TM::ld(&v.x[j]); };
  for (int I = clo + threadIdx.x; I < chi; I += tm.stride()) {
    int X0, Y0, Z0;
    level_coords(nC, I, X0, Y0, Z0);
    float sum = 0.f;
    for (int dz = 0; dz < (dim >= 3 ? 2 : 1); ++dz)
      for (int dy = 0; dy < (dim >= 2 ? 2 : 1); ++dy)
#pragma unroll
        for (int dx = 0; dx < 2; ++dx) {
          const int fx = 2 * X0 + dx, fy = 2 * Y0 + dy, fz = 2 * Z0 + dz;
          if (fx < n[0] && fy < n[1] && fz < n[2]) {
            const int c = fx + n[0] * (fy + n[1] * fz);
            sum += TM::ld(&v.b[c]) - level_apply(v.dg, v.cx, v.cy, v.cz, at, n, dim, c, nc);
          }
        }
    vc.b[I] = sum;
  }
  tm.sync();
}

// Coarsest level: x = Ainv b (dense).
template <class TM>
__device__ void vcoarsest(const MGArgs& A, const InstMG& m, const LevelView& v, TM& tm) {
  const int nc = (int)m.nc[m.levels - 1];
  int lo, hi;
  tm.range(nc, lo, hi);
  const float* inv = A.cinv + m.cinv_off;
  for (int i = lo + threadIdx.x; i < hi; i += tm.stride()) {
    float sum = 0.f;
    for (int j = 0; j < nc; ++j) sum += inv[i * nc + j] * TM::ld(&v.b[j]);
    v.x[i] = sum;
  }
  tm.sync();
}

// Upward half on level l: prolongation of the level l + 1 correction vc.x (injection scaled by
// alpha, the prolonged iterate formed where it is read), then two sweeps: v.x to v.t to v.x. The
// caller's next barrier orders the last one.
template <class TM>
__device__ void vup(const MGArgs& A, const InstMG& m, int l, const LevelView& v, const LevelView& vc, TM& tm) {
  const int nc = (int)m.nc[l], dim = m.dim;
  const int n[3] = {m.n[l][0], m.n[l][1], m.n[l][2]};
  const int nC[3] = {m.n[l + 1][0], m.n[l + 1][1], m.n[l + 1][2]};
  level_each(tm, l, nc, v.t, [&](int i) {
    int X0, Y0, Z0;
    level_coords(n, i, X0, Y0, Z0);
    const int I = (X0 >> 1) + nC[0] * ((Y0 >> 1) + nC[1] * (Z0 >> 1));
    const float ui = fmaf(A.alpha, TM::ld(&vc.x[I]), TM::ld(&v.x[i]));
    const float au = level_apply_prolonged<TM>(v.dg, v.cx, v.cy, v.cz, v.x, vc.x, A.alpha, n, nC, dim, i, X0, Y0, Z0);
    return ui + A.omega * (TM::ld(&v.b[i]) - au) * v.dinv[i];
  });
  tm.sync();
  auto at = [&](int j) { return TM::ld(&v.t[j]); };
  level_each(tm, l, nc, v.x, [&](int i) {
    const float ax = level_apply(v.dg, v.cx, v.cy, v.cz, at, n, dim, i, nc);
    return at(i) + A.omega * (TM::ld(&v.b[i]) - ax) * v.dinv[i];
  });
}

// First level of an instance that the first block handles alone (the coarsest at the latest).
__host__ __device__ __forceinline__ int solo_level(const InstMG& m, long long solo_cells) {
  int ls = 0;
  while (ls < m.levels - 1 && m.nc[ls] > solo_cells) ++ls;
  return ls;
}

// One V-cycle: lx = M^{-1} lb on the finest level. The caller's last barrier ordered lb; its
// next one orders lx. The team shares the levels above solo_level; the first block copies that
// level's right-hand side into its shared memory, runs the rest of the cycle there, and writes
// the level's correction back for the team.
template <class TM>
__device__ void vcycle(const MGArgs& A, const InstMG& m, TM& tm, float* smem) {
  const int L = m.levels;
  const int ls = solo_level(m, TM::solo_cells);
  SoloTeam solo;
  solo.nt = min((int)blockDim.x, ((int)m.nc[ls] + 31) & ~31);
  for (int l = 0; l < ls; ++l) vdown(A, m, l, global_view(A, m, l), global_view(A, m, l + 1), tm);
  if (tm.rank == 0 && (int)threadIdx.x < solo.nt) {
    const LevelView top = solo_view(A, m, ls, ls, smem);
    const float* gb = A.lb + m.off[ls];
    for (int i = threadIdx.x; i < m.nc[ls]; i += solo.nt) top.b[i] = __ldcg(&gb[i]);
    solo.sync();
    for (int l = ls; l < L - 1; ++l) vdown(A, m, l, solo_view(A, m, l, ls, smem), solo_view(A, m, l + 1, ls, smem), solo);
    vcoarsest(A, m, solo_view(A, m, L - 1, ls, smem), solo);
    for (int l = L - 2; l >= ls; --l) {
      vup(A, m, l, solo_view(A, m, l, ls, smem), solo_view(A, m, l + 1, ls, smem), solo);
      solo.sync();
    }
    float* gx = A.lx + m.off[ls];
    for (int i = threadIdx.x; i < m.nc[ls]; i += solo.nt) gx[i] = top.x[i];
  }
  tm.sync();
  for (int l = ls - 1; l >= 0; --l) {
    vup(A, m, l, global_view(A, m, l), global_view(A, m, l + 1), tm);
    if (l > 0) tm.sync();
  }
}

// The right-hand side of one cell (global index g), and the solution's use: see CorrectionIO.
__device__ __forceinline__ double correction_rhs(const MGArgs& A, const InstDesc& in, long long g) {
  const CorrectionIO& o = A.io;
  if (o.at) {
    const double h = o.at[g] + o.g[g];
    o.half_out[g] = h;
    return h - o.lam[g];
  }
  const long long base = in.bc_off + (g - in.cell_off);
  double r = 0.0;
  for (int b = 0; b < A.nb; ++b) r += o.R[base + (long long)b * in.ncells];
  return (r - o.T[g] * o.Vm[g]) / in.V;
}

__device__ __forceinline__ void correction_apply(const MGArgs& A, int k, long long g, double x) {
  const CorrectionIO& o = A.io;
  if (o.at) o.out[g] = o.half_out[g] + o.theta_m[g] * x;
  else o.out[g] = o.half[g] + o.theta[k] * x;
}

// A x of the FP64 fine operator for the cell at instance index i (global index g); V is read
// through L2 (other blocks of the team wrote it).
__device__ __forceinline__ double fine_apply(const MGArgs& A, const InstMG& m, const double* V, int i, long long g) {
  const int n = (int)m.nc[0], sy = m.n[0][0], sz = m.n[0][0] * m.n[0][1];
  double q = A.diag[g] * __ldcg(&V[g]);
  if (i + 1 < n) q -= A.cx[g] * __ldcg(&V[g + 1]);
  if (i >= 1) q -= A.cx[g - 1] * __ldcg(&V[g - 1]);
  if (m.dim >= 2) {
    if (i + sy < n) q -= A.cy[g] * __ldcg(&V[g + sy]);
    if (i >= sy) q -= A.cy[g - sy] * __ldcg(&V[g - sy]);
  }
  if (m.dim >= 3) {
    if (i + sz < n) q -= A.cz[g] * __ldcg(&V[g + sz]);
    if (i >= sz) q -= A.cz[g - sz] * __ldcg(&V[g - sz]);
  }
  return q;
}

// ---- Fast diagonalization (Lynch, Rice and Thomas 1964) for separable operators ----
// With A = Tx (x) I + I (x) Ty, Tx = Qx Lx Qx^T and Ty = Qy Ly Qy^T, and the right-hand side
// as an ny x nx matrix S (row j = the cells of y-row j), A X = S is solved by
//   X = Qy [(Qy^T S Qx) ./ (ly_j + lx_i)] Qx^T,
// four dense products of FP32 matrices (nx, ny <= FD_MAX_N). The rows j are split over the
// team's blocks. The solve runs inside FP64 iterative refinement: the solution is accumulated in
// FP64 and its residual S - A X is formed with the FP64 operator, until it meets rtol.
//
// A block has few rows (8 of a 192 x 192 grid on 24 blocks), so a product is bound by the L2 reads
// of its right operand, which every block reads whole: it streams through shared memory in
// chunks of its rows (asynchronous copies, two chunks ahead), and each warp multiplies units of
// 32 columns x 4 rows. The terms of an output are added one after the other, in ascending order,
// or, where both axes have at most FD_QUAD_N cells, in ascending groups of four with the last of a
// group first: a product does not depend on how many blocks share the instance (the order of the
// residual norm's FP64 sum does).
constexpr int FD_RB = 8;         // rows of a strip at most
constexpr int FD_QUAD_N = 128;
constexpr int FD_CHUNK = 8192;   // floats of a chunk (a multiple of 4 rows, 4 at least: FD_MAX_N <= 2048)
constexpr int FD_BUFS = 3;
constexpr int FD_UNITS = 4;      // units of a warp at most: 2 x FD_MAX_N / 32 over FD_NT / 32 warps
static_assert(2 * (FD_MAX_N / 32) <= FD_UNITS * (FD_NT / 32), "units per warp");

// Floats of a left operand's row in shared memory (zero beyond the true length; 16-byte rows).
__host__ __device__ constexpr int fd_row(int nmax) { return ((nmax + 3) & ~3) + 4; }
// Shared memory: chunks, two left operands kept over the passes, one between products.
__host__ __device__ constexpr size_t fd_smem_floats(int nmax) { return FD_BUFS * FD_CHUNK + 3 * (size_t)FD_RB * fd_row(nmax); }

// out(r, i, sum over k < K of L[r][k] R(k, i)) for r < nr (at most FD_RB), i < N; L in shared memory
// (rows ls apart), R in global memory (K x N, 16-byte aligned, written before the last barrier).
template <bool QUAD, class FE>
__device__ __forceinline__ void strip_product(const float* L, int ls, const float* R, int K, int N, int nr, float* stage,
                                              FE out) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int KC = (FD_CHUNK / N) & ~3, nch = (K + KC - 1) / KC;
  auto fetch = [&](int c) {
    if (c < nch) {
      const int beg = c * KC * N, end = min(K, (c + 1) * KC) * N;
      float* dst = stage + (c % FD_BUFS) * FD_CHUNK;
      const int n4 = (end - beg) >> 2;
      for (int e = threadIdx.x; e < n4; e += FD_NT) {
        const unsigned d = (unsigned)__cvta_generic_to_shared(dst + 4 * e);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(R + beg + 4 * e) : "memory");
      }
      if (c == nch - 1) {  // the last few floats, and zeros up to a multiple of four rows
        const int all = ((K - c * KC + 3) & ~3) * N;
        for (int e = 4 * n4 + threadIdx.x; e < all; e += FD_NT) dst[e] = beg + e < end ? __ldcg(&R[beg + e]) : 0.f;
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int ncb = (N + 31) / 32, units = ncb * ((nr + 3) / 4);
  int col[FD_UNITS];
  const float* row[FD_UNITS];
  float acc[FD_UNITS][4];
#pragma unroll
  for (int u = 0; u < FD_UNITS; ++u) {
    const int unit = min(warp + u * (FD_NT / 32), units - 1), g = unit / ncb;
    col[u] = min((unit - g * ncb) * 32 + lane, N - 1);  // beyond N: the last column's, not used
    row[u] = L + 4 * g * ls;
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[u][r] = 0.f;
  }
#pragma unroll
  for (int c = 0; c < FD_BUFS - 1; ++c) fetch(c);
  for (int c = 0; c < nch; ++c) {
    asm volatile("cp.async.wait_group %0;" ::"n"(FD_BUFS - 2) : "memory");
    __syncthreads();  // chunk c is there; chunk c - 1 is read
    fetch(c + FD_BUFS - 1);
    const float* buf = stage + (c % FD_BUFS) * FD_CHUNK;
    const int k0 = c * KC, kn = min(KC, (K - k0 + 3) & ~3);
#pragma unroll
    for (int u = 0; u < FD_UNITS; ++u) {
      if (warp + u * (FD_NT / 32) >= units) break;
      const float* bc = buf + col[u];
#pragma unroll 2
      for (int k = 0; k < kn; k += 4) {
        const float b0 = bc[k * N], b1 = bc[(k + 1) * N], b2 = bc[(k + 2) * N], b3 = bc[(k + 3) * N];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const float4 l = *reinterpret_cast<const float4*>(row[u] + r * ls + k0 + k);
          if (QUAD) acc[u][r] = fmaf(l.x, b0, fmaf(l.y, b1, fmaf(l.z, b2, fmaf(l.w, b3, acc[u][r]))));
          else acc[u][r] = fmaf(l.w, b3, fmaf(l.z, b2, fmaf(l.y, b1, fmaf(l.x, b0, acc[u][r]))));
        }
      }
    }
  }
#pragma unroll
  for (int u = 0; u < FD_UNITS; ++u) {
    const int unit = warp + u * (FD_NT / 32);
    if (unit >= units) break;
    const int g = unit / ncb, i = (unit - g * ncb) * 32 + lane;
    if (i < N) {
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (4 * g + r < nr) out(4 * g + r, i, acc[u][r]);
    }
  }
  __syncthreads();
}

// Solves the instance's correction by fast diagonalization with FP64 refinement (at most
// MG32_PASSES_FD passes); returns the passes taken, or -1 if rtol was not met.
template <bool QUAD>
__device__ int fd_solve(const MGArgs& A, int k, const InstMG& m, Team& tm, double* sh, float* smem) {
  const int nx = m.fnx, ny = m.fny, ls = fd_row(max(nx, ny));
  const long long off = m.cell_off;
  const int rows = (((ny + 3) / 4 + tm.size - 1) / tm.size) * 4;  // whole groups of four
  const int j0 = min(ny, tm.rank * rows), j1 = min(ny, j0 + rows);
  const int lo = j0 * nx, hi = j1 * nx;  // this block's cells
  const float* Qx = A.fq + m.qx_off;
  const float* QxT = A.fq + m.qxt_off;
  const float* Qy = A.fq + m.qy_off;
  const float* lx = A.flam + m.lx_off;
  const float* ly = A.flam + m.ly_off;
  float* Sf = A.lt + m.off[0];  // scaled residual (FP32)
  float* T2 = A.lx + m.off[0];  // (Qy^T S Qx) ./ (ly + lx)
  float* stage = smem;
  float* qc = stage + FD_BUFS * FD_CHUNK;  // rows of Qy^T: Qy(k, j)
  float* qr = qc + FD_RB * ls;             // rows of Qy: Qy(j, k)
  float* mid = qr + FD_RB * ls;            // rows between the two products of a half
  const bool keep = rows <= FD_RB;         // one strip: its left operands stay over the passes
  for (int e = threadIdx.x; e < 3 * FD_RB * ls; e += FD_NT) qc[e] = 0.f;
  __syncthreads();
  auto load_qc = [&](int jb, int nr) {
    for (int e = threadIdx.x; e < ny * FD_RB; e += FD_NT) {
      const int kk = e / FD_RB, r = e - kk * FD_RB;
      if (r < nr) qc[r * ls + kk] = __ldg(&Qy[(long long)kk * ny + jb + r]);
    }
  };
  auto load_qr = [&](int jb, int nr) {
    for (int e = threadIdx.x; e < ny * nr; e += FD_NT) {
      const int r = e / ny, kk = e - r * ny;
      qr[r * ls + kk] = __ldg(&Qy[(long long)(jb + r) * ny + kk]);
    }
  };
  if (keep) {
    load_qc(j0, j1 - j0);
    load_qr(j0, j1 - j0);
  }
  double v[1] = {0.0};
  for (int c = lo + threadIdx.x; c < hi; c += FD_NT) {
    const double b = correction_rhs(A, A.inst[k], off + c);
    A.rhs[off + c] = b;
    A.X[off + c] = 0.0;
    A.Z[off + c] = b;  // FP64 residual
    v[0] += b * b;
  }
  tm.sum<1>(v, sh);
  const double bb = v[0], tol2 = A.rtol * A.rtol * bb;
  int passes = bb == 0.0 ? 0 : -1;
  double rr = bb;
  for (int pass = 1; passes < 0 && pass <= MG32_PASSES_FD && pass <= A.maxit; ++pass) {
    const double rn = sqrt(rr), sc = 1.0 / rn;
    for (int c = lo + threadIdx.x; c < hi; c += FD_NT) Sf[c] = (float)(A.Z[off + c] * sc);
    tm.sync();
    // T2 = (Qy^T S Qx) ./ (ly_j + lx_i), strip by strip
    for (int jb = j0; jb < j1; jb += FD_RB) {
      const int nr = min(FD_RB, j1 - jb);
      if (!keep) load_qc(jb, nr);
      strip_product<QUAD>(qc, ls, Sf, ny, nx, nr, stage, [&](int r, int i, float x) { mid[r * ls + i] = x; });
      strip_product<QUAD>(mid, ls, Qx, nx, nx, nr, stage, [&](int r, int i, float x) {
        const int j = jb + r;
        T2[j * nx + i] = x / (ly[j] + lx[i]);
      });
    }
    tm.sync();
    // the correction (Qy T2) Qx^T added to the FP64 solution (scaled back)
    for (int jb = j0; jb < j1; jb += FD_RB) {
      const int nr = min(FD_RB, j1 - jb);
      if (!keep) load_qr(jb, nr);
      strip_product<QUAD>(qr, ls, T2, ny, nx, nr, stage, [&](int r, int i, float x) { mid[r * ls + i] = x; });
      strip_product<QUAD>(mid, ls, QxT, nx, nx, nr, stage,
                          [&](int r, int i, float x) { A.X[off + (jb + r) * nx + i] += (double)x * rn; });
    }
    tm.sync();
    // FP64 residual of the FP64 solution
    v[0] = 0.0;
    for (int c = lo + threadIdx.x; c < hi; c += FD_NT) {
      const double r = A.rhs[off + c] - fine_apply(A, m, A.X, c, off + c);
      A.Z[off + c] = r;
      v[0] += r * r;
    }
    tm.sum<1>(v, sh);  // also orders the residual's writes before the next pass
    rr = v[0];
    if (rr <= tol2) passes = pass;
  }
  for (int c = lo + threadIdx.x; c < hi; c += FD_NT) correction_apply(A, k, off + c, A.X[off + c]);
  return passes;
}

// The team of this block; its barrier starts from arrivals of 0.
__device__ __forceinline__ Team block_team(const MGArgs& A, TeamDesc& d) {
  const int t = A.block_team[blockIdx.x];
  d = A.teams[t];
  Team tm;
  tm.rank = (int)blockIdx.x - d.first_block;
  tm.size = d.size;
  tm.ctr = A.bar + 2 * t;
  tm.target = 0;
  tm.err = A.err;
  tm.slots = A.slots + 4 * (size_t)d.first_block;
  tm.buf = 0;
  tm.dead = false;
  return tm;
}

__device__ __forceinline__ ClusterTeam block_cluster(const MGArgs& A, TeamDesc& d, double* slots) {
  d = A.teams[A.block_team[blockIdx.x]];
  ClusterTeam tm;
  tm.rank = (int)blockIdx.x - d.first_block;
  tm.size = d.size;
  tm.slots = slots;
  tm.buf = 0;
  return tm;
}

// No block leaves while another may read its shared memory.
__device__ __forceinline__ void leave_team(ClusterTeam& tm) { tm.sync(); }

// The last block of a team to leave sets its barrier back for the next launch.
__device__ __forceinline__ void leave_team(Team& tm) {
  if (tm.size == 1) return;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    if (atomicAdd(tm.ctr + 1, 1u) == (unsigned)tm.size - 1u) {
      tm.ctr[0] = 0u;
      tm.ctr[1] = 0u;
    }
  }
}

__global__ void __launch_bounds__(FD_NT, 1) fd_kernel(MGArgs A) {
  __shared__ double sh[66];
  extern __shared__ float4 smem4[];
  float* smem = reinterpret_cast<float*>(smem4);
  TeamDesc d;
  Team tm = block_team(A, d);
  for (int q = d.inst_beg; q < d.inst_end; ++q) {
    const int k = A.order[q];
    const InstMG& m = A.mg[k];
    const int passes = m.fnx <= FD_QUAD_N && m.fny <= FD_QUAD_N ? fd_solve<true>(A, k, m, tm, sh, smem)
                                                                 : fd_solve<false>(A, k, m, tm, sh, smem);
    if (tm.rank == 0 && threadIdx.x == 0) A.iters_out[k] = tm.dead ? -1 : passes;
    __syncthreads();
  }
  leave_team(tm);
}

// FP64 iterates, for tolerances near FP32's rounding.
template <class TM>
__device__ __forceinline__ void mgpcg(const MGArgs& A, TM& tm, const TeamDesc& d, double* sh, float* mg_smem) {
  for (int iq = d.inst_beg; iq < d.inst_end; ++iq) {
    const int k = A.order[iq];
    const InstMG& m = A.mg[k];
    const long long off = m.cell_off;
    const Units un((int)m.nc[0], tm);
    float* b32 = A.lb + m.off[0];
    const float* x32 = A.lx + m.off[0];
    double v[1] = {0.0};
    // x = 0, r = b
    un.each([&](int i) {
      const double bi = correction_rhs(A, A.inst[k], off + i);
      A.X[off + i] = 0.0;
      A.Rr[off + i] = bi;
      b32[i] = (float)bi;
      v[0] += bi * bi;
    });
    tm.sum<1>(v, sh);
    const double bb = v[0];
    int it = 0;
    bool done = bb == 0.0;
    if (!done) {
      const double tol2 = A.rtol * A.rtol * bb;
      vcycle(A, m, tm, mg_smem);
      v[0] = 0.0;
      un.each([&](int i) {
        const double zi = (double)x32[i];
        A.P[off + i] = zi;
        v[0] += A.Rr[off + i] * zi;
      });
      tm.sum<1>(v, sh);  // also orders the P writes before the first product
      double rz = v[0];
      while (it < A.maxit && !tm.dead) {
        ++it;
        v[0] = 0.0;
        un.each([&](int i) {
          const double q = fine_apply(A, m, A.P, i, off + i);
          A.Q[off + i] = q;
          v[0] += __ldcg(&A.P[off + i]) * q;
        });
        tm.sum<1>(v, sh);
        const double alpha = rz / v[0];
        v[0] = 0.0;
        un.each([&](int i) {
          const long long g = off + i;
          A.X[g] += alpha * A.P[g];
          const double ri = A.Rr[g] - alpha * A.Q[g];
          A.Rr[g] = ri;
          b32[i] = (float)ri;
          v[0] += ri * ri;
        });
        tm.sum<1>(v, sh);
        if (v[0] <= tol2) {
          done = true;
          break;
        }
        vcycle(A, m, tm, mg_smem);
        // Flexible (Polak-Ribiere) beta = z_new . (r_new - r_old) / (z_old . r_old), with
        // r_new - r_old = -alpha q: robust to the FP32 preconditioner's rounding.
        double w[2] = {0.0, 0.0};
        un.each([&](int i) {
          const double zi = (double)x32[i];
          w[0] += A.Rr[off + i] * zi;
          w[1] += A.Q[off + i] * zi;
        });
        tm.sum<2>(w, sh);
        const double beta = -alpha * w[1] / rz;
        rz = w[0];
        un.each([&](int i) { A.P[off + i] = (double)x32[i] + beta * A.P[off + i]; });
        tm.sync();
      }
    }
    un.each([&](int i) { correction_apply(A, k, off + i, A.X[off + i]); });
    if (tm.rank == 0 && threadIdx.x == 0) A.iters_out[k] = done && !tm.dead ? it : -1;
    __syncthreads();
  }
  leave_team(tm);
}

// PCG with FP32 iterates for tolerances far above FP32's rounding (the correction is an
// inexact Newton step: its tolerance sets the cost, not the fixed point), inside FP64
// iterative refinement: the solution is accumulated in FP64 and its residual b - A x is
// formed and measured in FP64 with the FP64 operator; while that residual exceeds the
// tolerance (at most MG32_PASSES times) the FP32 PCG solves for the correction of that
// residual. Each pass scales its right-hand side to unit norm (so the FP32 sums neither
// underflow nor overflow); the stencil product uses the FP32 copy of the fine operator (the
// hierarchy's finest level); dot products are FP32 per lane of a unit and FP64 across them.
// On GB300 FP64 arithmetic issues on a narrow pipe, so FP64 iterates would lengthen every
// phase of the iteration; here FP64 enters once per pass. The finest level's right-hand side and
// iterate are the CG's residual and preconditioned residual themselves.
constexpr int MG32_PASSES = 4;

template <class TM>
__device__ __forceinline__ void mgpcg32(const MGArgs& A, float* V32, TM& tm, const TeamDesc& d, double* sh, float* mg_smem) {
  auto* st1 = reinterpret_cast<float(*)[32]>(mg_smem);
  auto* st2 = reinterpret_cast<float(*)[64]>(mg_smem);
  auto* st3 = reinterpret_cast<float(*)[96]>(mg_smem);
  for (int iq = d.inst_beg; iq < d.inst_end; ++iq) {
    const int k = A.order[iq];
    const InstMG& m = A.mg[k];
    const long long off = m.cell_off;
    const int n = (int)m.nc[0];
    const Units un(n, tm);
    float* R = A.lb + m.off[0];  // residual = the V-cycle's finest right-hand side
    float* Z = A.lx + m.off[0];  // preconditioned residual = its finest iterate
    float* X = V32 + 3 * off;
    float* P = X + n;
    float* Q = P + n;
    const float *dg = A.ldiag + m.off[0], *cx = A.lcx + m.off[0], *cy = A.lcy + m.off[0], *cz = A.lcz + m.off[0];
    const int nf[3] = {m.n[0][0], m.n[0][1], m.n[0][2]};
    double v[1] = {0.0};
    // x = 0, FP64 residual r = b
    un.each([&](int i) {
      const double bi = correction_rhs(A, A.inst[k], off + i);
      A.rhs[off + i] = bi;
      A.X[off + i] = 0.0;
      A.Z[off + i] = bi;
      v[0] += bi * bi;
    });
    tm.sum<1>(v, sh);
    const double bb = v[0];
    const double tol2 = A.rtol * A.rtol * bb;
    double rr = bb;  // FP64 squared norm of the FP64 residual
    int it = 0;
    bool done = bb == 0.0;
    for (int pass = 0; !done && pass < MG32_PASSES && it < A.maxit && !tm.dead; ++pass) {
      // FP32 PCG for A e = r (scaled to unit norm) to the relative tolerance the FP64 residual
      // still needs, at least the requested one and at most 1/2
      const double rn = sqrt(rr), sc = 1.0 / rn;
      const double rin = fmin(0.5, fmax(A.rtol, A.rtol * sqrt(bb) / rn));
      const double in2 = rin * rin;
      un.each([&](int i) {
        R[i] = (float)(A.Z[off + i] * sc);
        X[i] = 0.f;
      });
      tm.sync();
      vcycle(A, m, tm, mg_smem);
      un.dot<2, 1, 0, 1>(
          [&](int i, float(&x)[2]) {
            const float zi = __ldcg(&Z[i]);
            P[i] = zi;
            x[0] = R[i];
            x[1] = zi;
          },
          st2, v);
      tm.sum<1>(v, sh);  // also orders the P writes before the first product
      double rz = v[0];
      while (it < A.maxit && !tm.dead) {
        ++it;
        auto at = [&](int j) { return __ldcg(&P[j]); };
        un.dot<2, 1, 0, 1>(
            [&](int i, float(&x)[2]) {
              const float q = level_apply(dg, cx, cy, cz, at, nf, m.dim, i, n);
              Q[i] = q;
              x[0] = at(i);
              x[1] = q;
            },
            st2, v);
        tm.sum<1>(v, sh);
        const double alpha = rz / v[0];
        const float af = (float)alpha;
        un.dot<1, 1, 0, 0>(
            [&](int i, float(&x)[1]) {
              X[i] += af * P[i];
              const float ri = R[i] - af * Q[i];
              R[i] = ri;
              x[0] = ri;
            },
            st1, v);
        tm.sum<1>(v, sh);  // also orders the residual's writes before the V-cycle
        if (v[0] <= in2) break;
        vcycle(A, m, tm, mg_smem);
        // flexible (Polak-Ribiere) beta, as in the FP64 kernel
        double w[2];
        un.dot<3, 2, 0x10, 0x22>(
            [&](int i, float(&x)[3]) {
              x[0] = R[i];
              x[1] = Q[i];
              x[2] = __ldcg(&Z[i]);
            },
            st3, w);
        tm.sum<2>(w, sh);
        const double beta = -alpha * w[1] / rz;
        rz = w[0];
        const float bf = (float)beta;
        un.each([&](int i) { P[i] = __ldcg(&Z[i]) + bf * P[i]; });
        tm.sync();
      }
      // x += rn e in FP64, then the FP64 residual of x
      un.each([&](int i) { A.X[off + i] += (double)X[i] * rn; });
      tm.sync();
      v[0] = 0.0;
      un.each([&](int i) {
        const double r = A.rhs[off + i] - fine_apply(A, m, A.X, i, off + i);
        A.Z[off + i] = r;
        v[0] += r * r;
      });
      tm.sum<1>(v, sh);  // also orders the residual's writes before the next pass
      rr = v[0];
      done = rr <= tol2;
    }
    un.each([&](int i) { correction_apply(A, k, off + i, A.X[off + i]); });
    if (tm.rank == 0 && threadIdx.x == 0) A.iters_out[k] = done && !tm.dead ? it : -1;
    __syncthreads();
  }
  leave_team(tm);
}

// Shared memory: the levels the first block handles alone, or staged products.
__global__ void __launch_bounds__(MG_NT, 1) mgpcg_kernel(MGArgs A) {
  __shared__ double sh[66];
  extern __shared__ float mg_smem[];
  TeamDesc d;
  Team tm = block_team(A, d);
  mgpcg(A, tm, d, sh, mg_smem);
}
__global__ void __launch_bounds__(MG_NT, 1) mgpcg32_kernel(MGArgs A, float* V32) {
  __shared__ double sh[66];
  extern __shared__ float mg_smem[];
  TeamDesc d;
  Team tm = block_team(A, d);
  mgpcg32(A, V32, tm, d, sh, mg_smem);
}
__global__ void __launch_bounds__(MG_SMALL_NT, 1) mgpcg_cluster_kernel(MGArgs A) {
  __shared__ double sh[66], slots[4];
  extern __shared__ float mg_smem[];
  TeamDesc d;
  ClusterTeam tm = block_cluster(A, d, slots);
  mgpcg(A, tm, d, sh, mg_smem);
}
__global__ void __launch_bounds__(MG_SMALL_NT, 1) mgpcg32_cluster_kernel(MGArgs A, float* V32) {
  __shared__ double sh[66], slots[4];
  extern __shared__ float mg_smem[];
  TeamDesc d;
  ClusterTeam tm = block_cluster(A, d, slots);
  mgpcg32(A, V32, tm, d, sh, mg_smem);
}

// Tolerances from here up run the FP32 iterates.
constexpr double MG32_MIN_RTOL = 1e-5;

// Deals `blocks` blocks to the instances `which`, instance i in parts[i] equal parts of cost[i]: one
// team per instance while there are blocks enough (the instance whose blocks have most to do grows
// next, to the next size at which they have less; never more than parts[i]); else one-block teams
// that take the instances in turn, the costliest first to the team with the least to do.
static void plan_teams(const std::vector<int>& which, const std::vector<double>& cost, const std::vector<int>& parts,
                       int blocks, std::vector<TeamDesc>& teams, std::vector<int>& order, std::vector<int>& block_team) {
  const int n = (int)which.size();
  teams.clear();
  order.clear();
  block_team.clear();
  if (n == 0) return;
  if (n <= blocks) {
    std::vector<int> size(n, 1);
    auto per = [&](int i) { return (parts[i] + size[i] - 1) / size[i]; };
    for (int left = blocks - n; left > 0;) {
      int best = 0;
      for (int i = 1; i < n; ++i)
        if (per(i) * cost[i] > per(best) * cost[best]) best = i;
      if (per(best) == 1) break;
      const int next = (parts[best] + per(best) - 2) / (per(best) - 1);  // one part less per block
      if (next - size[best] > left) break;
      left -= next - size[best];
      size[best] = next;
    }
    for (int i = 0; i < n; ++i) {
      teams.push_back({(int)block_team.size(), size[i], i, i + 1});
      order.push_back(which[i]);
      for (int b = 0; b < size[i]; ++b) block_team.push_back(i);
    }
    return;
  }
  std::vector<int> by(n);
  for (int i = 0; i < n; ++i) by[i] = i;
  std::stable_sort(by.begin(), by.end(), [&](int a, int b) { return cost[a] * parts[a] > cost[b] * parts[b]; });
  std::vector<std::vector<int>> list(blocks);
  std::vector<double> load(blocks, 0.0);
  for (int i : by) {
    const int t = (int)(std::min_element(load.begin(), load.end()) - load.begin());
    list[t].push_back(which[i]);
    load[t] += cost[i] * parts[i];
  }
  for (int t = 0; t < blocks; ++t) {
    teams.push_back({t, 1, (int)order.size(), (int)(order.size() + list[t].size())});
    order.insert(order.end(), list[t].begin(), list[t].end());
    block_team.push_back(t);
  }
}

// Cluster teams that run at once on an otherwise idle device (0 where a cluster does not fit).
static cudaError_t cluster_teams(const Ctx* c, size_t smem, int* most) {
  const void* f[2] = {(const void*)mgpcg_cluster_kernel, (const void*)mgpcg32_cluster_kernel};
  *most = 0;
  for (int i = 0; i < 2; ++i) {
    cudaError_t e = allow_shared(f[i], c->smem_optin);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(MG_CLUSTER, 1, 1);
    cfg.blockDim = dim3(MG_SMALL_NT, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = MG_CLUSTER;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if ((e = cudaOccupancyMaxActiveClusters(&n, f[i], &cfg)) != cudaSuccess) return e;
    *most = i == 0 ? n : std::min(*most, n);
  }
  return cudaSuccess;
}

// Uploads the team plans of the two kernels (separable operators, the others) and sets the
// kernels' shared memory.
cudaError_t configure_mgpcg(Ctx* c, const std::vector<InstMG>& h_mg) {
  for (int kind = 0; kind < 2; ++kind) {  // 0: multigrid CG, 1: fast diagonalization
    TeamPlan& p = c->team_plan[kind];
    std::vector<int> which, parts;
    std::vector<double> cost;
    size_t smem = 0;
    for (int k = 0; k < (int)h_mg.size(); ++k) {
      const InstMG& m = h_mg[k];
      if ((m.direct != 0) != (kind == 1)) continue;
      which.push_back(k);
      if (kind == 1) {  // parts: groups of four rows, by the terms of their products
        parts.push_back((m.fny + 3) / 4);
        cost.push_back((double)m.fnx * (m.fnx + m.fny));
        smem = std::max(smem, fd_smem_floats(std::max(m.fnx, m.fny)) * sizeof(float));
      } else {
        // parts: units, by their steps; no more blocks than give every warp a step, and one for
        // small instances
        const long long chunk = (m.nc[0] + MG_RANKS - 1) / MG_RANKS, steps = (chunk + 32 * MG_WARPS - 1) / (32 * MG_WARPS);
        const long long units = (long long)MG_RANKS << range_units_log(chunk);
        const int most =
            m.nc[0] <= MG_SMALL_CELLS ? 1 : (int)std::max<long long>(1, std::min(units, units * steps / (MG_NT / 32)));
        parts.push_back(most);
        cost.push_back((double)steps * units / most);
        size_t cells = 0;
        for (int l = solo_level(m, Team::solo_cells); l < m.levels; ++l) cells += (size_t)m.nc[l];
        smem = std::max(std::max(smem, 3 * cells * sizeof(float)), (size_t)MG_STAGE * 96 * sizeof(float));
      }
    }
    p.blocks = 0;
    p.smem = smem;
    p.threads = kind ? FD_NT : MG_NT;
    p.cluster = false;
    if (which.empty()) continue;
    cudaError_t e;
    long long largest = 0;
    for (int k : which) largest = std::max<long long>(largest, h_mg[k].nc[0]);
    if (kind == 0 && largest > MG_CLUSTER_FROM && largest <= MG_CLUSTER_CELLS) {
      int most = 0;
      if ((e = cluster_teams(c, smem, &most)) != cudaSuccess) return e;
      p.cluster = (int)which.size() <= most;
    }
    if (kind == 0 && (p.cluster || largest <= MG_SMALL_CELLS)) p.threads = MG_SMALL_NT;
    const void* f[2] = {kind ? (const void*)fd_kernel : (const void*)mgpcg_kernel,
                        kind ? (const void*)fd_kernel : (const void*)mgpcg32_kernel};
    for (const void* q : f) {
      if ((e = allow_shared(q, c->smem_optin)) != cudaSuccess) return e;
      int nb = 0;
      if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, q, kind ? FD_NT : MG_NT, smem)) != cudaSuccess) return e;
      if (nb < 1) return cudaErrorLaunchOutOfResources;
    }
    std::vector<TeamDesc> teams;
    std::vector<int> order, block_team;
    if (p.cluster) {
      order = which;
      for (int i = 0; i < (int)which.size(); ++i) {
        teams.push_back({MG_CLUSTER * i, MG_CLUSTER, i, i + 1});
        block_team.insert(block_team.end(), MG_CLUSTER, i);
      }
    } else {
      plan_teams(which, cost, parts, c->sm_count, teams, order, block_team);
    }
    p.blocks = (int)block_team.size();
    // one buffer: partial sums and barrier words (zero), then the plan
    const size_t at_bar = 4 * block_team.size() * sizeof(double), at_teams = at_bar + 2 * teams.size() * sizeof(unsigned),
                 at_order = at_teams + teams.size() * sizeof(TeamDesc), at_block = at_order + order.size() * sizeof(int);
    std::vector<char> h(at_block + block_team.size() * sizeof(int), 0);
    std::memcpy(h.data() + at_teams, teams.data(), teams.size() * sizeof(TeamDesc));
    std::memcpy(h.data() + at_order, order.data(), order.size() * sizeof(int));
    std::memcpy(h.data() + at_block, block_team.data(), block_team.size() * sizeof(int));
    if ((e = cudaMalloc((void**)&p.d_buf, h.size())) != cudaSuccess) return e;
    if ((e = cudaMemcpy(p.d_buf, h.data(), h.size(), cudaMemcpyHostToDevice)) != cudaSuccess) return e;
    p.d_slots = reinterpret_cast<double*>(p.d_buf);
    p.d_bar = reinterpret_cast<unsigned*>(p.d_buf + at_bar);
    p.d_teams = p.d_buf + at_teams;
    p.d_order = reinterpret_cast<int*>(p.d_buf + at_order);
    p.d_block_team = reinterpret_cast<int*>(p.d_buf + at_block);
  }
  return cudaSuccess;
}

static cudaError_t launch_correction(const Ctx* c, const CorrectionIO& io, cudaStream_t s) {
  MGArgs a;
  a.mg = c->d_mg;
  a.inst = c->d_inst;
  a.nb = c->nb;
  a.err = c->d_err;
  a.io = io;
  a.diag = c->d_diag;
  a.cx = c->d_cx;
  a.cy = c->d_cy;
  a.cz = c->d_cz;
  a.ldiag = c->d_mg_diag;
  a.ldiag_inv = c->d_mg_dinv;
  a.lcx = c->d_mg_cx;
  a.lcy = c->d_mg_cy;
  a.lcz = c->d_mg_cz;
  a.cinv = c->d_mg_cinv;
  a.fq = c->d_fd_q;
  a.flam = c->d_fd_lam;
  a.lb = c->d_mg_b;
  a.lx = c->d_mg_x;
  a.lt = c->d_mg_t;
  a.rhs = c->d_work;
  a.X = c->d_pcg;
  a.Rr = c->d_pcg + c->total_cells;
  a.P = c->d_pcg + 2 * c->total_cells;
  a.Q = c->d_pcg + 3 * c->total_cells;
  a.Z = c->d_pcg + 4 * c->total_cells;
  a.rtol = c->opt.cg_rtol;
  a.maxit = c->opt.cg_maxit;
  a.iters_out = c->d_pcg_iters;
  a.alpha = 1.8f;
  a.omega = 0.8f;
  for (int kind = 0; kind < 2; ++kind) {
    const TeamPlan& p = c->team_plan[kind];
    if (p.blocks == 0) continue;
    a.teams = static_cast<const TeamDesc*>(p.d_teams);
    a.block_team = p.d_block_team;
    a.order = p.d_order;
    a.bar = p.d_bar;
    a.slots = p.d_slots;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.blocks, 1, 1);
    cfg.blockDim = dim3(p.threads, 1, 1);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    if (p.cluster) {
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = MG_CLUSTER;
      attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    } else {
      attr[0].id = cudaLaunchAttributeCooperative;  // the blocks of a team wait for one another
      attr[0].val.cooperative = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaError_t e;
    if (kind == 1) {
      e = cudaLaunchKernelEx(&cfg, fd_kernel, a);
    } else if (c->opt.cg_rtol >= MG32_MIN_RTOL) {
      // FP32 x, p, q in the space of the FP64 r and p (2 n doubles = 4 n floats >= 3 n floats);
      // the FP64 residual of the refinement in that of z
      float* v32 = reinterpret_cast<float*>(c->d_pcg + c->total_cells);
      e = cudaLaunchKernelEx(&cfg, p.cluster ? mgpcg32_cluster_kernel : mgpcg32_kernel, a, v32);
    } else {
      e = cudaLaunchKernelEx(&cfg, p.cluster ? mgpcg_cluster_kernel : mgpcg_kernel, a);
    }
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// T_half += theta dT with dT solving the diffusion problem for the Newton source
// s = (sum_b R_b - T_n V m) / V (absorbed minus emitted power density).
cudaError_t launch_newton(const Ctx* c, const double* T_n, double* T_half, const double* R, cudaStream_t s) {
  CorrectionIO io = {};
  io.R = R;
  io.T = T_n;
  io.Vm = c->d_Vm;
  io.theta = c->d_theta;
  io.half = T_half;
  io.out = T_half;
  return launch_correction(c, io, s);
}

// Adjoint correction: half = at + g, out = half + theta m D^{-1}(half - lam) (transpose of the
// forward step T += theta D^{-1} m (T_half - T); D symmetric).
cudaError_t launch_adjoint_correction(const Ctx* c, const double* at, const double* g, const double* lam, double* half,
                                      double* out, cudaStream_t s) {
  CorrectionIO io = {};
  io.at = at;
  io.g = g;
  io.lam = lam;
  io.theta_m = c->d_theta_m;
  io.half_out = half;
  io.out = out;
  return launch_correction(c, io, s);
}

}  // namespace iugkp
