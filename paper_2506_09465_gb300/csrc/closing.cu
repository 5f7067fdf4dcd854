// What surrounds the trace of a sweep: one pass before it (every buffer cleared, emitter weights
// and their largest per instance) and the passes after it (W scaled, the faces that are not
// tallied, the power entering and leaving through the walls). Each is one launch where its data
// allow it: on small grids these passes, not the trace, set the time of a sweep.
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"

namespace iugkp {

namespace {

// Instance holding entry j of a [band][cell] array: the last one whose bc_off is at or before j.
__device__ __forceinline__ int bc_instance(const InstDesc* inst, int n_inst, long long j) {
  int lo = 0, hi = n_inst - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (inst[mid].bc_off <= j) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ int cell_instance(const InstDesc* inst, int n_inst, long long g) {
  int lo = 0, hi = n_inst - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (inst[mid].cell_off <= g) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Before the trace. Every block clears its share of the list; the claim counters take their
// start values; blocks [0, P.wmax_blocks) also compute their emitters' weights (group g has blocks
// [bpre[g], bpre[g + 1]), in proportion to its emitters) and the largest |weight| of each, and
// the last of those blocks to finish reduces them per instance. The largest is taken on the bit
// patterns of the magnitudes (integer compares: the FP64 pipe is narrow), NaN left out.
__global__ void __launch_bounds__(256) prologue_kernel(SweepArgs A, PrologueArgs P) {
  const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
  for (int s = 0; s < P.n_clear; ++s)
    for (long long i = tid; i < P.words[s]; i += step) P.clear[s][i] = 0ull;
  if (P.next)
    for (long long k = tid; k < P.n_inst; k += step) P.next[k] = P.next_from[k];
  if ((int)blockIdx.x >= P.wmax_blocks) return;
  __shared__ unsigned long long sh[8];
  __shared__ bool last;
  int gi = 0;
  {
    int hi = A.n_groups - 1;  // the last group whose first block is at or before this one
    while (gi < hi) {
      const int mid = (gi + hi + 1) >> 1;
      if (P.bpre[mid] <= (int)blockIdx.x) gi = mid;
      else hi = mid - 1;
    }
  }
  const Group G = A.groups[gi];
  const int by = (int)blockIdx.x - P.bpre[gi], ny = P.bpre[gi + 1] - P.bpre[gi];
  const InstDesc& in = A.inst[G.inst];
  unsigned long long m = 0;
  auto take = [&](double w) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(w) & 0x7fffffffffffffffull;
    if (b <= 0x7ff0000000000000ull && b > m) m = b;
  };
  if (G.kind == 0) {
    const double* coef = A.coef + in.bc_off + (long long)G.band * in.ncells;
    double* out = A.wemit + in.bc_off + (long long)G.band * in.ncells;
    const double* T = A.T + in.cell_off;
    const double* sft = A.srcshift ? A.srcshift + in.cell_off : nullptr;
    const int ncells = in.ncells, hop = ny * 256;
    for (int e0 = by * 256 + threadIdx.x; e0 < ncells; e0 += 4 * hop) {
      double t[4], c[4], d[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {  // the loads of four emitters in flight
        const int e = e0 + u * hop;
        t[u] = e < ncells ? __ldg(&T[e]) : 0.0;
        c[u] = e < ncells ? __ldg(&coef[e]) : 0.0;
        d[u] = sft && e < ncells ? __ldg(&sft[e]) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e0 + u * hop;
        if (e >= ncells) break;
        const double w = c[u] * (sft ? t[u] + d[u] : t[u]);
        out[e] = w;  // the weight of every particle of this emitter
        take(w);
      }
    }
  } else {
    const int wl = G.kind - 1;
    const double wc = A.wcoef[((long long)G.inst * A.nb + G.band) * 6 + wl];
    const double* tf = A.wallTf + in.bface_off + in.wface_off[wl];
    for (int j = by * 256 + threadIdx.x; j < G.n_emitters; j += ny * 256) take(wc * tf[j]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long t = __shfl_down_sync(0xffffffffu, m, o);
    m = t > m ? t : m;
  }
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) m = sh[w] > m ? sh[w] : m;
    P.wpart[blockIdx.x] = m;
    __threadfence();
    last = atomicAdd(P.ticket, 1u) == (unsigned)P.wmax_blocks - 1u;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int k = threadIdx.x; k < P.n_inst; k += 256) P.wmax[k] = 0ull;
  if (threadIdx.x == 0) *P.ticket = 0u;
  __syncthreads();
  for (int b = threadIdx.x; b < P.wmax_blocks; b += 256) {
    int g = 0, hi = A.n_groups - 1;
    while (g < hi) {
      const int mid = (g + hi + 1) >> 1;
      if (P.bpre[mid] <= b) g = mid;
      else hi = mid - 1;
    }
    const unsigned long long v = __ldcg(&P.wpart[b]);
    if (v) atomicMax(&P.wmax[A.groups[g].inst], v);
  }
}

// After the trace, per cell over its bands: absorbed minus emitted power sum_b R_b - V m T_emit
// (T_emit = T + Q/m) into bal, and the candidate estimator W = sum of w tau_maj over candidates
// (Sec. 3.2): the trace sums w per (band, cell), or nothing in a band whose every candidate is
// real (there W = tau_maj R). One read of R for both.
__device__ __forceinline__ void finish_cell(const SweepArgs& A, int n_inst, const double* Vm, double* bal, long long g) {
  const int k = cell_instance(A.inst, n_inst, g);
  const InstDesc& in = A.inst[k];
  const long long j0 = in.bc_off + (g - in.cell_off);
  double r = 0.0;
  for (int b0 = 0; b0 < A.nb; b0 += 8) {
    double x[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)  // the loads of eight bands in flight
      x[u] = b0 + u < A.nb ? __ldg(&A.R[j0 + (long long)(b0 + u) * in.ncells]) : 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if (b0 + u >= A.nb) break;
      r += x[u];
      if (A.W) {
        const long long j = j0 + (long long)(b0 + u) * in.ncells;
        const int kb = k * A.nb + b0 + u;
        A.W[j] = (__ldg(&A.all_real[kb]) ? x[u] : A.W[j]) * __ldg(&A.taumaj[kb]);
      }
    }
  }
  if (bal) {
    double te = A.T[g];
    if (A.srcshift) te += A.srcshift[g];
    bal[g] = r - Vm[g] * te;
  }
}

__device__ __forceinline__ void scale_entry(const SweepArgs& A, int k, long long j) {
  const int kb = A.nb == 1 ? k : k * A.nb + (int)((j - A.inst[k].bc_off) / A.inst[k].ncells);
  A.W[j] = (A.all_real[kb] ? A.R[j] : A.W[j]) * A.taumaj[kb];
}

// Faces of wall w = 2a + side of an instance, enumerated as j1 + n(o1) j2 (o1 = (a+1)%3,
// o2 = (a+2)%3); returns the face index within the instance.
__device__ __forceinline__ long long wall_face(const InstDesc& in, int a, int side, int j) {
  const int n0 = in.n[0], n1 = in.n[1], n2 = in.n[2];
  if (a == 0) {
    const int j1 = j % n1, j2 = j / n1;
    return in.fax_off[0] + (side ? n0 : 0) + (long long)(n0 + 1) * (j1 + (long long)n1 * j2);
  }
  if (a == 1) {
    const int j1 = j % n2, j2 = j / n2;
    return in.fax_off[1] + j2 + (long long)n0 * ((side ? n1 : 0) + (long long)(n1 + 1) * j1);
  }
  const int j1 = j % n0, j2 = j / n0;
  return in.fax_off[2] + j1 + (long long)n0 * (j2 + (long long)n1 * (side ? n2 : 0));
}

__device__ __forceinline__ int wall_faces(const InstDesc& in, int a) {
  return in.n[(a + 1) % 3] * in.n[(a + 2) % 3];
}

// One block: the power entering through the faces of wall wl of instance k (N_w particles of
// weight C_b v_b A T_w / (4 N_w) per face and band) added to F when `emit`, and the wall's
// absorbed power (fixed-order reduction) when `absorbed`: the sum of its faces as tallied, before
// the emission enters them; or, where the emission is in them already, that emission plus the
// outward net flux (a difference, to the rounding of the emission).
__device__ void wall_block(const SweepArgs& A, const double* wall_unit, int k, int wl, bool emit, bool absorbed) {
  __shared__ double sh[8], shT[8];
  const int a = wl >> 1, side = wl & 1;
  const InstDesc& in = A.inst[k];
  const int nf = wall_faces(in, a);
  const double u = wall_unit[k * 6 + wl];
  const double* tf = A.wallTf + in.bface_off + in.wface_off[wl];
  double sum = 0.0, tsum = 0.0;
  for (int j = threadIdx.x; j < nf; j += blockDim.x) {
    const long long f = in.face_off + wall_face(in, a, side, j);
    const double v = __ldcg(&A.F[f]);
    sum += v;
    if (emit) {
      const double e = u * tf[j];
      if (e != 0.0) A.F[f] = v + (side ? -e : e);
    }
    tsum += tf[j];
  }
  if (!absorbed) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sum += __shfl_down_sync(0xffffffffu, sum, o);
    tsum += __shfl_down_sync(0xffffffffu, tsum, o);
  }
  __syncthreads();  // the previous wall's sums are read
  if ((threadIdx.x & 31) == 0) {
    sh[threadIdx.x >> 5] = sum;
    shT[threadIdx.x >> 5] = tsum;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0, ts = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      t += sh[w];
      ts += shT[w];
    }
    A.wall[in.wall_off + wl] = (emit ? 0.0 : u * ts) + (side ? t : -t);
  }
}

// After a trace that tallied every face (the staged sweep in 1D, the filtered FP64 sweep in 2D and 3D):
// blocks [0, roles) take the walls (one wall each; in 1D one instance each, after its faces are formed
// from the fixed-point sums Fi and the FP64 sums Fx), the others scale W.
__global__ void __launch_bounds__(256) close_tallied_kernel(SweepArgs A, int n_inst, const double* wall_unit,
                                                            const long long* Fi, const double* Fx, const double* wmax,
                                                            long long total_bc, int roles) {
  if ((int)blockIdx.x < roles) {
    if (A.dim == 1) {
      const int k = blockIdx.x;
      const InstDesc& in = A.inst[k];
      const double qs = wmax[k] / WIN_SCALE;
      for (long long f = in.face_off + threadIdx.x; f < in.face_off + in.nfaces; f += 256)
        A.F[f] = Fi[f] ? fma((double)Fi[f], qs, Fx[f]) : Fx[f];
      __threadfence_block();
      __syncthreads();
      for (int wl = 0; wl < 2; ++wl) wall_block(A, wall_unit, k, wl, true, A.wall != nullptr);
    } else {
      const int k = blockIdx.x / (2 * A.dim);
      wall_block(A, wall_unit, k, blockIdx.x - k * 2 * A.dim, true, A.wall != nullptr);
    }
    return;
  }
  if (!A.W) return;
  const long long step = (long long)(gridDim.x - roles) * blockDim.x;
  for (long long j = ((long long)blockIdx.x - roles) * blockDim.x + threadIdx.x; j < total_bc; j += step)
    scale_entry(A, bc_instance(A.inst, n_inst, j), j);
}

// After the filtered FP64 sweep in 1D: blocks [0, roles) add to every face (which holds the replayed
// particles' crossings) the nodes above its leaf, over the copies; a boundary face is its wall's
// absorbed power then, and the wall's emission enters it. The others scale W.
__global__ void __launch_bounds__(256) close_runs_kernel(SweepArgs A, int n_inst, const double* wall_unit, const double* node,
                                                         long long stride, int copies, long long total_faces,
                                                         long long total_bc, int roles) {
  if ((int)blockIdx.x < roles) {
    // eight lanes per face, lane q on the tree's levels q, q + 8, .. above the leaf: one or two L2
    // round trips in a row, not one per level (51 faces: 6 us less)
    const int q = threadIdx.x & 7;
    for (long long g0 = blockIdx.x * 32ll; g0 < total_faces; g0 += roles * 32ll) {
      const long long g = g0 + (threadIdx.x >> 3);
      const bool ok = g < total_faces;
      int k = 0;
      for (int hi = n_inst - 1; k < hi;) {  // the last instance whose faces start at or before g
        const int mid = (k + hi + 1) >> 1;
        if (A.inst[mid].face_off <= g) k = mid;
        else hi = mid - 1;
      }
      const InstDesc& in = A.inst[k];
      const int n = (int)in.nfaces, f = (int)(g - in.face_off);
      const double* t = node + 2 * in.face_off;
      double v = 0.0;
      for (unsigned i = ok ? (unsigned)(f + n) >> q : 0u; i; i >>= 8) {
        double x[EXACT_NODE_COPIES];
#pragma unroll
        for (int c = 0; c < EXACT_NODE_COPIES; ++c)  // the loads of all copies in flight
          x[c] = c < copies ? __ldcg(&t[c * stride + i]) : 0.0;
#pragma unroll
        for (int c = 0; c < EXACT_NODE_COPIES; ++c) v += x[c];
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (!ok || q != 0) continue;
      v += A.F[g];
      const int wl = f == 0 ? 0 : (f == n - 1 ? 1 : -1);
      if (wl >= 0) {
        if (A.wall) A.wall[in.wall_off + wl] = wl ? v : 0.0 - v;
        const double e = wall_unit[k * 6 + wl] * A.wallTf[in.bface_off + in.wface_off[wl]];
        if (e != 0.0) v += wl ? -e : e;
      }
      A.F[g] = v;
    }
    return;
  }
  if (!A.W) return;
  const long long step = (long long)(gridDim.x - roles) * blockDim.x;
  for (long long j = ((long long)blockIdx.x - roles) * blockDim.x + threadIdx.x; j < total_bc; j += step)
    scale_entry(A, bc_instance(A.inst, n_inst, j), j);
}

// Blocks [0, roles): emission through the walls (3D: all but the high z-wall, whose faces are
// derived); the others: one thread per cell (finish_cell).
__global__ void __launch_bounds__(256) finish_cells_kernel(SweepArgs A, int n_inst, long long total, const double* Vm,
                                                           const double* wall_unit, double* bal, int roles) {
  if ((int)blockIdx.x < roles) {
    const int k = blockIdx.x / (2 * A.dim - 1);
    wall_block(A, wall_unit, k, blockIdx.x - k * (2 * A.dim - 1), true, false);
    return;
  }
  const long long step = (long long)(gridDim.x - roles) * blockDim.x;
  for (long long g = ((long long)blockIdx.x - roles) * blockDim.x + threadIdx.x; g < total; g += step)
    finish_cell(A, n_inst, Vm, bal, g);
}

// 3D, faces normal to z from per-cell conservation:
// F[k+1] = F[k] + (net inflow through the other axes' faces of cell k) - (R_k - S_k), starting
// from the tallied low face (bal = R - S from finish_cell).
// Block: 32 adjacent columns x DERIVE_SEG segments (one warp per segment, so loads are
// coalesced across columns). Each thread sums its segment's increments, the segments'
// offsets follow from a prefix over the block's shared sums, then each thread writes its
// segment's running values.
constexpr int DERIVE_SEG = 8;

__device__ __forceinline__ double column_step(const InstDesc& in, const double* bal, const double* Fi, long long c) {
  const int n0 = in.n[0], n1 = in.n[1];
  const long long row = c / n0;  // x-face index of the cell's low face = c + row
  const int cz = (int)(c / ((long long)n0 * n1));
  const long long fy = in.fax_off[1] + c + (long long)n0 * cz;
  const double inflow = Fi[in.fax_off[0] + c + row] - Fi[in.fax_off[0] + c + row + 1] + (Fi[fy] - Fi[fy + n0]);
  return inflow - bal[in.cell_off + c];
}

__global__ void __launch_bounds__(32 * DERIVE_SEG) derive_z_kernel(const InstDesc* inst, int n_inst, const double* bal,
                                                                   double* F) {
  __shared__ double segsum[DERIVE_SEG][32];
  const int k = blockIdx.y;
  if (k >= n_inst) return;
  const InstDesc& in = inst[k];
  const int n0 = in.n[0], n1 = in.n[1], nlast = in.n[2];
  const int ncol = in.ncells / nlast;
  double* Fi = F + in.face_off;
  const int lane = threadIdx.x & 31, seg = threadIdx.x >> 5;
  const int seglen = (nlast + DERIVE_SEG - 1) / DERIVE_SEG;
  const int k0 = seg * seglen, k1 = min(nlast, k0 + seglen);
  for (int cbase = blockIdx.x * 32; cbase < ncol; cbase += gridDim.x * 32) {
    const int col = cbase + lane;
    const bool ok = col < ncol;
    const int ix = ok ? col % n0 : 0, iy = ok ? col / n0 : 0;
    const long long stride = (long long)n0 * n1, base_cell = ix + (long long)n0 * iy;
    double part = 0.0;
    if (ok)
      for (int kk = k0; kk < k1; ++kk) part += column_step(in, bal, Fi, base_cell + kk * stride);
    segsum[seg][lane] = part;
    __syncthreads();
    if (ok) {
      // low boundary face of this column, then the segments below this one
      double acc = Fi[in.fax_off[2] + base_cell];
      for (int sg = 0; sg < seg; ++sg) acc += segsum[sg][lane];
      for (int kk = k0; kk < k1; ++kk) {
        const long long c = base_cell + kk * stride;
        acc += column_step(in, bal, Fi, c);
        Fi[in.fax_off[2] + c + stride] = acc;
      }
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(256) wall_absorbed_kernel(SweepArgs A, const double* wall_unit) {
  wall_block(A, wall_unit, blockIdx.y, blockIdx.x, false, true);
}

// After the 2D staged trace: every face of the caller's F in one launch, from the tallies the
// trace made (Fi, fixed-point sums in units of q = w_max / WIN_SCALE; Fx, FP64 sums of the replayed
// particles; GX, exits through the low walls of untallied axes).
//
// Instances without the two-group tallies: faces normal to x are tallied; faces normal to y
// follow column by column from the bottom up from per-cell conservation:
//   F[j+1] = F[j] + (X[i,j] - X[i+1,j]) - (R - S)_c.
// Two-group instances: the faces each group did not tally follow from that group's power
// balance in every cell. x-group, column i, faces normal to y from the bottom up:
//   G[j+1] = G[j] + (X[i,j] - X[i+1,j]) - ((R - S)_c - D_y,c),
// starting from the x-group's net flux through the bottom face (its exits there plus its
// share of the wall's emission, the whole emission minus the y-group's); X are the x-group's
// tallied faces plus its share of the emission on the x-walls. y-group, row j, faces
// normal to x from the left:
//   H[i+1] = H[i] + (Y[i,j] - Y[i,j+1]) - D_y,c,
// starting from its exits through the left wall and its emission there; Y are its tallied
// faces plus its emission on the y-walls. Every face is its tallied group's sum + the other
// group's derived flux + the tallied group's share of the wall emission.
//
// One warp per line (columns write the faces normal to y, rows those normal to x), prefix sums
// over chunks of 32 cells in a fixed order; F is only written. The last line block of an
// instance to finish sums its walls' absorbed power. Blocks beyond the lines scale W (one band;
// with more bands finish_cells_kernel has done it, and bal holds the balances).
__global__ void __launch_bounds__(256) close_2d_kernel(SweepArgs A, Close2D C) {
  const int k = blockIdx.y;
  const InstDesc& in = A.inst[k];
  const int n0 = in.n[0], n1 = in.n[1];
  const int nline_blocks = (n0 + n1 + 7) / 8;
  if ((int)blockIdx.x >= C.line_blocks) {  // W
    const long long end = in.bc_off + (long long)A.nb * in.ncells, step = (long long)(gridDim.x - C.line_blocks) * 256;
    for (long long j = in.bc_off + ((long long)blockIdx.x - C.line_blocks) * 256 + threadIdx.x; j < end; j += step)
      scale_entry(A, k, j);
    return;
  }
  if ((int)blockIdx.x >= nline_blocks) return;
  const bool two = C.window[k].x == 0 && (long long)C.window[k].y == in.nfaces;
  const double qs = C.wmax[k] / WIN_SCALE;
  const int line = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const long long* Fi = C.Fi + in.face_off;
  const double* Fx = C.Fx + in.face_off;
  double* F = A.F + in.face_off;
  const long long fax1 = in.fax_off[1];
  const double* ey = C.EY + in.bface_off;
  const double* tf = A.wallTf + in.bface_off;
  const double* dy = C.DY + in.cell_off;
  auto tallied = [&](long long f) { return Fi[f] ? fma((double)Fi[f], qs, Fx[f]) : Fx[f]; };
  // the exit tally of boundary face j, summed over the copies of GX
  auto gx = [&](long long j) {
    double t = 0.0;
#pragma unroll
    for (int r = 0; r < GX_COPIES; ++r) t += C.GX[r * C.gx_stride + in.bface_off + j];
    return t;
  };
  // signed flux of the whole emission of wall wl through its face j
  auto etot = [&](int wl, int j) {
    const double e = C.wall_unit[k * 6 + wl] * tf[in.wface_off[wl] + j];
    return (wl & 1) ? -e : e;
  };
  // emission through the x-walls that belongs to the tallied faces normal to x
  auto ex = [&](int wl, int j) { return etot(wl, j) - (two ? ey[in.wface_off[wl] + j] : 0.0); };
  if (line < n0) {
    const int i = line;
    double acc = gx(in.wface_off[2] + i) + etot(2, i) - (two ? ey[in.wface_off[2] + i] : 0.0);
    if (lane == 0) F[fax1 + i] = acc + (two ? tallied(fax1 + i) + ey[in.wface_off[2] + i] : Fx[fax1 + i]);
    if (!two) acc += Fx[fax1 + i];
    for (int j0 = 0; j0 < n1; j0 += 32) {
      const int j = j0 + lane;
      double v = 0.0;
      if (j < n1) {
        const long long c = i + (long long)n0 * j;
        const long long fl = c + j;  // x-face (i, j)
        double left = tallied(fl), right = tallied(fl + 1);
        if (i == 0) left += ex(0, j);
        if (i == n0 - 1) right += ex(1, j);
        double bal;
        if (C.bal) {
          bal = C.bal[in.cell_off + c];
        } else {
          double te = A.T[in.cell_off + c];
          if (A.srcshift) te += A.srcshift[in.cell_off + c];
          bal = A.R[in.bc_off + c] - C.Vm[in.cell_off + c] * te;
        }
        if (two) bal -= dy[c];
        v = (left - right) - bal;
      }
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const double t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
      }
      if (j < n1) {
        const long long f = fax1 + i + (long long)n0 * (j + 1);
        double x = acc + v;
        if (two) {
          x += tallied(f);
          if (j == n1 - 1) x += ey[in.wface_off[3] + i];
        }
        F[f] = x;
      }
      acc += __shfl_sync(0xffffffffu, v, 31);
    }
  } else if (line < n0 + n1) {
    const int j = line - n0;
    const long long row = (long long)(n0 + 1) * j;
    double acc = two ? gx(in.wface_off[0] + j) + ey[in.wface_off[0] + j] : 0.0;
    if (lane == 0) F[row] = acc + tallied(row) + ex(0, j);
    for (int ib = 0; ib < n0; ib += 32) {
      const int i = ib + lane;
      double v = 0.0;
      if (two && i < n0) {
        const long long c = i + (long long)n0 * j;
        double bot = tallied(fax1 + c), top = tallied(fax1 + c + n0);
        if (j == 0) bot += ey[in.wface_off[2] + i];
        if (j == n1 - 1) top += ey[in.wface_off[3] + i];
        v = (bot - top) - dy[c];
      }
      if (two) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const double t = __shfl_up_sync(0xffffffffu, v, o);
          if (lane >= o) v += t;
        }
      }
      if (i < n0) {
        double x = acc + v + tallied(row + i + 1);
        if (i == n0 - 1) x += ex(1, j);
        F[row + i + 1] = x;
      }
      if (two) acc += __shfl_sync(0xffffffffu, v, 31);
    }
  }
  if (!A.wall) return;
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&C.ticket[k], 1u) == (unsigned)nline_blocks - 1u;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (threadIdx.x == 0) C.ticket[k] = 0u;
  // absorbed power of each wall, one warp per wall: its emission plus the outward net flux
  const int wl = threadIdx.x >> 5;
  if (wl >= 4) return;
  const int a = wl >> 1, side = wl & 1, nf = a == 0 ? n1 : n0;
  double sum = 0.0, tsum = 0.0;
  for (int j0 = lane; j0 < nf; j0 += 128) {
    double v[4], t[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {  // the loads of four faces in flight
      const int j = j0 + 32 * u;
      const long long f = a == 0 ? (side ? n0 : 0) + (long long)(n0 + 1) * j : fax1 + j + (long long)n0 * (side ? n1 : 0);
      v[u] = j < nf ? __ldcg(&F[f]) : 0.0;
      t[u] = j < nf ? tf[in.wface_off[wl] + j] : 0.0;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      sum += v[u];
      tsum += t[u];
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sum += __shfl_down_sync(0xffffffffu, sum, o);
    tsum += __shfl_down_sync(0xffffffffu, tsum, o);
  }
  if (lane == 0) A.wall[in.wall_off + wl] = C.wall_unit[k * 6 + wl] * tsum + (side ? sum : -sum);
}

}  // namespace

cudaError_t launch_prologue(const Ctx* c, const SweepArgs& a, const PrologueArgs& P, cudaStream_t s) {
  long long words = 0;
  for (int i = 0; i < P.n_clear; ++i) words += P.words[i];
  const long long want = std::min<long long>((words + 1023) / 1024, 8ll * c->sm_count);
  const unsigned blocks = (unsigned)std::max<long long>(1, std::max<long long>(want, P.wmax_blocks));
  prologue_kernel<<<blocks, 256, 0, s>>>(a, P);
  return cudaGetLastError();
}

static unsigned cell_blocks(const Ctx* c, long long n) {
  return (unsigned)std::max<long long>(1, std::min<long long>((n + 255) / 256, 8ll * c->sm_count));
}

cudaError_t launch_close_tallied(const Ctx* c, const SweepArgs& a, cudaStream_t s) {
  const long long bc = (long long)c->nb * c->total_cells;
  const unsigned extra = a.W ? cell_blocks(c, bc) : 0;
  if (c->dim == 1 && a.F) {
    const int roles = (int)cell_blocks(c, 8 * c->total_faces);
    close_runs_kernel<<<roles + extra, 256, 0, s>>>(a, c->n_inst, c->d_wall_unit, c->d_nodes, 2 * c->total_faces,
                                                    c->node_copies, c->total_faces, bc, roles);
    return cudaGetLastError();
  }
  const int roles = a.F ? 2 * c->dim * c->n_inst : 0;
  if (roles + extra == 0) return cudaSuccess;
  close_tallied_kernel<<<roles + extra, 256, 0, s>>>(a, c->n_inst, c->d_wall_unit, nullptr, nullptr, nullptr, bc, roles);
  return cudaGetLastError();
}

cudaError_t launch_close_1d(const Ctx* c, const SweepArgs& a, cudaStream_t s) {
  const long long bc = (long long)c->nb * c->total_cells;
  const int roles = a.F ? c->n_inst : 0;
  const unsigned extra = a.W ? cell_blocks(c, bc) : 0;
  if (roles + extra == 0) return cudaSuccess;
  close_tallied_kernel<<<roles + extra, 256, 0, s>>>(a, c->n_inst, c->d_wall_unit, c->d_Fi, c->d_Fx,
                                                     reinterpret_cast<const double*>(c->d_wmax), bc, roles);
  return cudaGetLastError();
}

cudaError_t launch_close_3d(const Ctx* c, const SweepArgs& a, cudaStream_t s) {
  const int roles = a.F ? (2 * c->dim - 1) * c->n_inst : 0;
  if (!a.F && !a.W) return cudaSuccess;
  // the balance per cell goes into the correction solve's scratch (free until the Newton step,
  // which runs after the sweep on the same stream)
  finish_cells_kernel<<<roles + cell_blocks(c, c->total_cells), 256, 0, s>>>(
      a, c->n_inst, c->total_cells, c->d_Vm, c->d_wall_unit, a.F ? c->d_work : nullptr, roles);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || !a.F) return e;
  long long maxcol = 0;
  for (const InstDesc& in : c->h_inst) maxcol = std::max<long long>(maxcol, in.ncells / in.n[2]);
  dim3 grid((unsigned)std::min<long long>((maxcol + 31) / 32, 4096), (unsigned)c->n_inst);
  derive_z_kernel<<<grid, 32 * DERIVE_SEG, 0, s>>>(c->d_inst, c->n_inst, c->d_work, a.F);
  if ((e = cudaGetLastError()) != cudaSuccess || !a.wall) return e;
  wall_absorbed_kernel<<<dim3(2 * c->dim, c->n_inst), 256, 0, s>>>(a, c->d_wall_unit);
  return cudaGetLastError();
}

cudaError_t launch_close_2d(const Ctx* c, const SweepArgs& a, cudaStream_t s) {
  if (!a.F && !a.W) return cudaSuccess;
  cudaError_t e;
  const bool bands = c->nb > 1;
  if (bands || !a.F) {
    finish_cells_kernel<<<cell_blocks(c, c->total_cells), 256, 0, s>>>(a, c->n_inst, c->total_cells, c->d_Vm,
                                                                      c->d_wall_unit, a.F ? c->d_work : nullptr, 0);
    if ((e = cudaGetLastError()) != cudaSuccess || !a.F) return e;
  }
  Close2D C;
  C.window = c->d_window;
  C.wmax = reinterpret_cast<const double*>(c->d_wmax);
  C.Fi = c->d_Fi;
  C.Fx = c->d_Fx;
  C.bal = bands ? c->d_work : nullptr;
  C.Vm = c->d_Vm;
  C.wall_unit = c->d_wall_unit;
  C.DY = c->d_DY;
  C.EY = c->d_EY;
  C.GX = c->d_GX;
  C.gx_stride = c->total_bfaces;
  C.ticket = c->d_ticket + 1;
  long long lines = 0, cells = 0;
  for (const InstDesc& in : c->h_inst) {
    lines = std::max<long long>(lines, in.n[0] + in.n[1]);
    cells = std::max<long long>(cells, in.ncells);
  }
  C.line_blocks = (int)((lines + 7) / 8);
  const unsigned extra = a.W && !bands ? (unsigned)std::min<long long>((cells + 1023) / 1024, 64) : 0;
  close_2d_kernel<<<dim3(C.line_blocks + extra, (unsigned)c->n_inst), 256, 0, s>>>(a, C);
  return cudaGetLastError();
}

}  // namespace iugkp
