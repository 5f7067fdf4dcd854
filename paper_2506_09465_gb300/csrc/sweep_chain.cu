// Fast forward sweep in 3D: long chains of null candidates (arXiv 2506.09465 Sec. 3.2). Same
// particles, draws, decisions and tallies as the 1D / 2D staged sweep (sweep_staged.cu): FP32 along
// the straight segment where a bound shows the decision to be the FP64 walk's, the rest queued
// for the FP64 replay; x- and y-faces tallied with global FP64 atomics, the faces normal to z
// derived from per-cell conservation.
//
// A two-material box has ten candidates per particle, from one on the thick side to sixty on the
// thin side. When a lane walked, tallied and re-emitted by itself, 13 of 32 lanes were active (23.9
// ms for four boxes up to 64^3, 1.05e8 particles, 1.07e9 candidates). Here a warp runs three phases,
// each with nearly all lanes at work (25 of 32), that hand particles on through lists in shared
// memory (15.4 ms; the ratios of both candidates of a step in flight at once took it from 20.9; now
// bound by the latency of those loads and of the draws, and by the L2's atomics, 1.4e11 of at most
// 2.1e11 per second):
//   emit   32 particles at once; those that were walking wait;
//   walk   two candidates per step, from one Philox block; idle lanes take waiting particles;
//   end    32 ended particles at once: faces crossed, then their face items shared out.
#include <cuda_runtime.h>

#include "device.cuh"
#include "internal.h"
#include "landing.cuh"
#include "segment.cuh"
#include "staged.h"
#include "walk32.cuh"

namespace iugkp {

namespace {

// A warp's lists, one word per lane and field (lanes side by side: no bank conflicts). 8256 bytes,
// so that 20 warps leave the L1 92 KB for the acceptance ratios.
constexpr int RDY_F = 17;  // waiting: xi, s, cell coordinates, D, eD, particle, emission id, q, next pair, w
constexpr int END_F = 11;  // ended: xi, s, cell, end cell (wall: -1 - candidates), particle, w
constexpr int CHAIN_LISTS = 64;  // x- and y-faces of the particles of 32 lanes
struct ChainLists {
  int4 tab[CHAIN_LISTS * 3];  // item lists of the ended particles (parameters)
  unsigned rdy[RDY_F][31];    // (an idle lane makes the others wait)
  unsigned end[END_F][64];
  int lst[CHAIN_LISTS + 1];   // starts of the item lists
};

// Where a candidate lies. The positions of landing.cuh with twice the bound of the face counts of
// segment.cuh (plus the positions' own error, an eighth of it): away from the faces of every
// axis the cell and the side of every wall are what those counts give; closer (a few in 10^3), the
// counts themselves decide (`near`).
struct Spot {
  bool out, near;
};
enum { SPOT_IN = 0, SPOT_OUT, SPOT_NEAR };
__device__ __forceinline__ int spot_axis(float g, float D, float rel, float xi, int i, int n, Spot& p) {
  const float X = fmaf(g, D, xi), tol = fmaf(fabsf(g), rel, 2.f * TIE_REL);
  const float Y = __fadd_rn(X, FLOOR_MAGIC), off = X - (Y - FLOOR_MAGIC);  // from the nearest face
  const bool near = !(fabsf(off) > tol);                                   // a NaN too
  const int c = i + (__float_as_int(Y) - 0x4B400000) + (__float_as_int(off) >> 31);
  p.out |= !near && (unsigned)c >= (unsigned)n;
  p.near |= near;
  return c;
}

// axis_init with the distance to the first face rounded (not fused into what it is used for).
__device__ __forceinline__ void axis_rn(float s, float xi, float h, float& t, float& d, int& st) {
  st = s > 0.f ? 1 : -1;
  d = __fdividef(h, fabsf(s));
  t = __fmul_rn(s > 0.f ? 1.f - xi : xi, d);
}

}  // namespace

template <bool K32>
__global__ void __launch_bounds__(CHAIN_NT, 1) sweep_chain_kernel(SweepArgs A, StagedArgs S) {
  extern __shared__ int4 chain_smem[];
  __shared__ int s_inst;
  ChainLists& B = reinterpret_cast<ChainLists*>(chain_smem)[threadIdx.x >> 5];
  LCounts cnt;
#pragma unroll
  for (int k = 0; k < CNT_N; ++k) cnt.v[k] = 0;
  const int lane = threadIdx.x & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  const bool useF = A.F != nullptr;
  const bool useW = K32 ? S.W32 != nullptr : A.W != nullptr;
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
    const bool work = s_inst >= 0;
    __syncthreads();
    if (!work) continue;
    const InstDesc& in = A.inst[k];
    const int n0 = in.n[0], n1 = in.n[1], n2 = in.n[2], ncells = in.ncells;
    const int sy_cell = n0, sz_cell = n0 * n1;
    const long long bc_off = in.bc_off, face_off = in.face_off;
    const float ih0 = __frcp_rn(in.hf[0]), ih1 = __frcp_rn(in.hf[1]), ih2 = __frcp_rn(in.hf[2]);
    const uint32_t inst_id = in.inst_id;  // (the atomics would force reloads)
    const unsigned pend = (unsigned)S.inst_end[k];
    const int refill = S.refill > 0 ? S.refill : CHAIN_REFILL;
    unsigned rbeg = 0, rend = 0;  // this warp's range of particles
    bool exhausted = false;
    int nwait = 0, nend = 0, gi = 0;
    // the lane's particle: s its direction, g = s / h
    bool alive = false;
    float xi0 = 0.f, xi1 = 0.f, xi2 = 0.f, s0 = 0.f, s1 = 0.f, s2 = 0.f, g0 = 0.f, g1 = 0.f, g2 = 0.f, D = 0.f, eD = 0.f;
    int i0 = 0, i1 = 0, i2 = 0;
    unsigned pid = 0, id = 0;
    int pair = 0;      // its next pair of draws: block pair / 2, first or second half
    int band = 0, q = 0;
    float vtm = 0.f;   // v tau_maj of its band
    double w = 0.0;
    int kc = 0;        // candidates tallied
    int ecell = 0;     // cell of its real collision, -1: wall

    // The candidate at path length Dc (bound eDc): beyond a wall, near a face, or in `cell` with the
    // acceptance ratio ra (a load in flight).
    auto classify = [&](float Dc, float eDc, const float* ratio, bool all_real, int& cell, float& ra) -> int {
      const float rel = fmaf(Dc, 2.f * TIE_REL, 1.0625f * eDc);
      Spot p;
      p.out = p.near = false;
      const int p0 = spot_axis(g0, Dc, rel, xi0, i0, n0, p), p1 = spot_axis(g1, Dc, rel, xi1, i1, n1, p),
                p2 = spot_axis(g2, Dc, rel, xi2, i2, n2, p);
      cell = p0 + sy_cell * p1 + sz_cell * p2;
      ra = 1.f;
      if (!all_real) ra = __ldg(&ratio[p.out || p.near ? 0 : cell]);
      return p.out ? SPOT_OUT : (p.near ? SPOT_NEAR : SPOT_IN);
    };
    // Its outcome: 0 the particle goes on, 1 it has ended (ecell), 2 it is left to the FP64 replay.
    auto candidate = [&](int spot, int cell, float ra, uint32_t ub, long long bcbase, bool all_real) -> int {
      if (spot == SPOT_OUT) {
        ecell = -1;
        return 1;
      }
      int oc;
      if (spot == SPOT_IN) {
        const float ua = word_uniform<float>(ub);
        oc = fabsf(ua - ra) < TIE_ACC ? CAND_DEFER : (ua < ra ? CAND_REAL : CAND_NULL);
        if (all_real) oc = CAND_REAL;  // no draw was taken
      } else {
        PW f;
        f.i0 = i0;
        f.i1 = i1;
        f.i2 = i2;
        axis_rn(s0, xi0, in.hf[0], f.t0, f.d0, f.s0);
        axis_rn(s1, xi1, in.hf[1], f.t1, f.d1, f.s1);
        axis_rn(s2, xi2, in.hf[2], f.t2, f.d2, f.s2);
        f.D = D;
        f.tex = fminf(fminf(axis_exit(i0, f.s0, n0, f.t0, f.d0), axis_exit(i1, f.s1, n1, f.t1, f.d1)),
                      axis_exit(i2, f.s2, n2, f.t2, f.d2));
        const float base = fmaf(TIE_REL, D, eD);
        if (D - f.tex > base) {
          ecell = -1;
          return 1;
        }
        if (f.tex - D <= fmaf(TIE_REL, f.tex, eD)) return 2;
        bool close = false;
        int fb0, fb1, fb2;
        if (all_real) {
          fb0 = count_near(D, f.t0, f.d0, base, close);
          fb1 = count_near(D, f.t1, f.d1, base, close);
          fb2 = count_near(D, f.t2, f.d2, base, close);
        } else {
          fb0 = faces_before(D, f.t0, f.d0);
          fb1 = faces_before(D, f.t1, f.d1);
          fb2 = faces_before(D, f.t2, f.d2);
        }
        cell = clampi(i0 + f.s0 * fb0, n0) + sy_cell * clampi(i1 + f.s1 * fb1, n1) + sz_cell * clampi(i2 + f.s2 * fb2, n2);
        oc = candidate_outcome<3>(A, bcbase, ncells, f, base, fb0, fb1, fb2, cell, all_real, close, ub, n0, n1, n2,
                                  sy_cell, sz_cell);
      }
      if (oc == CAND_DEFER) return 2;
      ++kc;
      // W collects w here; the sweep scales it by tau_maj afterwards, and a band whose every
      // candidate is real takes W = tau_maj R there instead
      if (useW && !all_real) {
        if (K32) tally_k32(&S.W32[bcbase + cell], w);
        else atomicAdd(&A.W[bcbase + cell], w);
      }
      if (oc == CAND_NULL) return 0;
      cnt.v[CNT_REAL] += 1;
      if (K32) tally_k32(&S.R32[bcbase + cell], w);
      else atomicAdd(&A.R[bcbase + cell], w);
      ecell = cell;
      return 1;
    };
    // After a candidate: defers, or appends the lanes whose particles ended to the list.
    auto close_lane = [&](int res) {
      if (res != 0) {
        cnt.v[CNT_CANDIDATES] += kc;
        if (res == 2) defer_particle(S, pid, (unsigned)kc << 1);
        alive = false;
      }
      const unsigned m = __ballot_sync(0xffffffffu, res == 1);
      if (res == 1) {
        const int pos = nend + __popc(m & lt_mask);
        B.end[0][pos] = __float_as_uint(xi0);
        B.end[1][pos] = __float_as_uint(xi1);
        B.end[2][pos] = __float_as_uint(xi2);
        B.end[3][pos] = __float_as_uint(s0);
        B.end[4][pos] = __float_as_uint(s1);
        B.end[5][pos] = __float_as_uint(s2);
        B.end[6][pos] = (unsigned)(i0 + sy_cell * i1 + sz_cell * i2);
        B.end[7][pos] = (unsigned)(ecell >= 0 ? ecell : -1 - kc);
        B.end[8][pos] = pid;
        B.end[9][pos] = (unsigned)__double2loint(w);
        B.end[10][pos] = (unsigned)__double2hiint(w);
      }
      nend += __popc(m);
    };
    // Ended particles, the last 32 of the list: faces crossed, then the face items by the whole warp.
    auto end_phase = [&] {
      __syncwarp();
      const int first_rec = nend > 32 ? nend - 32 : 0, rec = first_rec + lane;
      int nx3 = 0, ny3 = 0;
      if (rec < nend) {
        float exi0 = __uint_as_float(B.end[0][rec]), exi1 = __uint_as_float(B.end[1][rec]),
              exi2 = __uint_as_float(B.end[2][rec]);
        PW f;
        const unsigned em = B.end[6][rec], emr = udiv(em, (unsigned)n0, S.mag_n0[k]);
        f.i2 = (int)udiv(emr, (unsigned)n1, S.mag_n1[k]);
        f.i1 = (int)emr - f.i2 * n1;
        f.i0 = (int)em - (int)emr * n0;
        axis_rn(__uint_as_float(B.end[3][rec]), exi0, in.hf[0], f.t0, f.d0, f.s0);
        axis_rn(__uint_as_float(B.end[4][rec]), exi1, in.hf[1], f.t1, f.d1, f.s1);
        axis_rn(__uint_as_float(B.end[5][rec]), exi2, in.hf[2], f.t2, f.d2, f.s2);
        const int ec = (int)B.end[7][rec];
        const double ew = __hiloint2double((int)B.end[10][rec], (int)B.end[9][rec]);
        const int m0 = faces_to_wall(f.i0, f.s0, n0), m1 = faces_to_wall(f.i1, f.s1, n1), m2 = faces_to_wall(f.i2, f.s2, n2);
        int c0, c1, c2, ex = -1;
        bool tie = false;
        if (ec >= 0) {  // the cells between the emission and the collision
          const int r = (int)udiv((unsigned)ec, (unsigned)n0, S.mag_n0[k]);
          const int e2 = (int)udiv((unsigned)r, (unsigned)n1, S.mag_n1[k]);
          c0 = abs(ec - r * n0 - f.i0);
          c1 = abs(r - e2 * n1 - f.i1);
          c2 = abs(e2 - f.i2);
        } else {
          // at a wall: on the exit axis the count is known; a count of the other axes within
          // rounding of the FP64 walk's (the segment leaves near a cell corner) defers the particle
          const float e0 = axis_exit(f.i0, f.s0, n0, f.t0, f.d0), e1 = axis_exit(f.i1, f.s1, n1, f.t1, f.d1),
                      e2 = axis_exit(f.i2, f.s2, n2, f.t2, f.d2);
          const float L = fminf(fminf(e0, e1), e2), bx = TIE_REL * L;
          ex = (e0 <= e1 && e0 <= e2) ? 0 : (e1 <= e2 ? 1 : 2);
          c0 = m0 - 1;
          c1 = m1 - 1;
          c2 = m2 - 1;
          if (ex != 0) c0 = min(count_near(L, f.t0, f.d0, bx, tie), m0 - 1);
          if (ex != 1) c1 = min(count_near(L, f.t1, f.d1, bx, tie), m1 - 1);
          if (ex != 2) c2 = min(count_near(L, f.t2, f.d2, bx, tie), m2 - 1);
        }
        if (tie) {
          defer_particle(S, B.end[8][rec], (unsigned)(-1 - ec) << 1);
        } else {
          if (ec < 0) cnt.v[CNT_WALL_EXITS] += 1;
          cnt.v[CNT_CROSSINGS] += c0 + c1 + c2;
          if (useF) {
            // faces normal to z: only the low boundary is tallied (the rest follow)
            if (ex == 2 && f.s2 < 0) {
              const long long fi = face_off + in.fax_off[2] + (f.i0 + f.s0 * c0) + (long long)n0 * (f.i1 + f.s1 * c1);
              if (K32) tally_k32(&S.F32[fi], -ew);
              else atomicAdd(&A.F[fi], -ew);
            }
            // Two item lists: the x-faces crossed (the wall face too when the particle leaves
            // through x) and the y-faces. Item j of the list along axis p is the face a0 + j sp + sq1
            // min(ceil(u1 + j r1), lim1) + sq2 min(ceil(u2 + j r2), lim2): the j-th face normal to p,
            // in the cell row and layer given by the faces of the other two axes crossed before it
            // (ceil((t_p + j d_p - t_q) / d_q) = ceil(u + j r), u = (t_p - t_q) / d_q, r = d_p / d_q).
            int4* tab = B.tab + 6 * lane;
            auto ur = [](float tp, float dp, float tq, float dq, float& u, float& r) {
              const bool flat = !(dq < INFINITY);
              u = flat ? -1.f : __fdividef(__fsub_rn(tp, tq), dq);
              r = flat ? 0.f : __fdividef(dp, dq);
            };
            const int sy_xf = n0 + 1, sz_xf = (n0 + 1) * n1, sz_yf = n0 * (n1 + 1);
            float u1, r1, u2, r2;
            nx3 = c0 + (ex == 0 ? 1 : 0);
            ny3 = c1 + (ex == 1 ? 1 : 0);
            ur(f.t0, f.d0, f.t1, f.d1, u1, r1);
            ur(f.t0, f.d0, f.t2, f.d2, u2, r2);
            double ws = f.s0 > 0 ? ew : -ew;
            tab[0] = make_int4((f.s0 > 0 ? f.i0 + 1 : f.i0) + sy_xf * f.i1 + sz_xf * f.i2, f.s0, f.s1 * sy_xf, m1 - 1);
            tab[1] = make_int4(f.s2 * sz_xf, m2 - 1, __float_as_int(u1), __float_as_int(r1));
            tab[2] = make_int4(__float_as_int(u2), __float_as_int(r2), __double2loint(ws), __double2hiint(ws));
            ur(f.t1, f.d1, f.t0, f.d0, u1, r1);
            ur(f.t1, f.d1, f.t2, f.d2, u2, r2);
            ws = f.s1 > 0 ? ew : -ew;
            tab[3] = make_int4((int)in.fax_off[1] + f.i0 + n0 * (f.s1 > 0 ? f.i1 + 1 : f.i1) + sz_yf * f.i2, f.s1 * n0,
                               f.s0, m0 - 1);
            tab[4] = make_int4(f.s2 * sz_yf, m2 - 1, __float_as_int(u1), __float_as_int(r1));
            tab[5] = make_int4(__float_as_int(u2), __float_as_int(r2), __double2loint(ws), __double2hiint(ws));
          }
        }
      }
      nend = first_rec;
      // the lists concatenated in order and cut into 32 equal contiguous chunks, one per lane
      int incl = nx3 + ny3;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      const int total = __shfl_sync(0xffffffffu, incl, 31);
      if (total > 0) {
        const int excl = incl - nx3 - ny3;
        B.lst[2 * lane] = excl;
        B.lst[2 * lane + 1] = excl + nx3;
        if (lane == 31) B.lst[CHAIN_LISTS] = total;
        __syncwarp();
        const int k0 = (int)(((long long)lane * total) >> 5), k1 = (int)(((long long)(lane + 1) * total) >> 5);
        if (k0 < k1) {
          int l = 0;  // the last list starting at or before k0
#pragma unroll
          for (int st = 32; st > 0; st >>= 1)
            if (B.lst[l + st] <= k0) l += st;
          int lbeg = B.lst[l], lend = B.lst[l + 1];
          int4 pa = B.tab[3 * l], pb = B.tab[3 * l + 1], pc = B.tab[3 * l + 2];
#pragma unroll 1
          for (int kk = k0; kk < k1; ++kk) {
            if (kk >= lend) {  // the next non-empty list
              do {
                ++l;
                lbeg = lend;
                lend = B.lst[l + 1];
              } while (lend <= kk);
              pa = B.tab[3 * l];
              pb = B.tab[3 * l + 1];
              pc = B.tab[3 * l + 2];
            }
            const float fk = small_int_float(kk - lbeg);
            const int face = pa.x + (kk - lbeg) * pa.y +
                             pa.z * min(ceil_count(fmaf(fk, __int_as_float(pb.w), __int_as_float(pb.z))), pa.w) +
                             pb.x * min(ceil_count(fmaf(fk, __int_as_float(pc.y), __int_as_float(pc.x))), pb.y);
            const double val = __hiloint2double(pc.w, pc.z);
            if (K32) tally_k32(&S.F32[face_off + face], val);
            else atomicAdd(&A.F[face_off + face], val);
          }
        }
      }
      __syncwarp();
    };

    for (;;) {
      const unsigned dead = __ballot_sync(0xffffffffu, !alive);
      const bool last = exhausted && nwait == 0 && dead == 0xffffffffu;
      if (nend >= 32 || (last && nend > 0)) {
        end_phase();
        continue;
      }
      if (last) break;
      int res = 0;
      uint32_t ub = 0;
      long long bcbase;
      bool all_real = false, second = false;  // second: the block's other pair is to come
      Stream st;
      if (__popc(dead) >= refill && nwait == 0 && !exhausted) {
        // ---- emit: the walking particles wait in the list, 32 new ones take their lanes ----
        if (rbeg == rend) {
          unsigned long long got = 0;
          if (lane == 0) got = atomicAdd(&S.inst_next[k], (unsigned long long)S.warp_grab);
          got = __shfl_sync(0xffffffffu, got, 0);
          if (got >= pend) {
            exhausted = true;
            continue;
          }
          rbeg = (unsigned)got;
          rend = (unsigned)min(got + (unsigned long long)S.warp_grab, (unsigned long long)pend);
        }
        if (alive) {
          const int pos = __popc(~dead & lt_mask);
          B.rdy[0][pos] = __float_as_uint(xi0);
          B.rdy[1][pos] = __float_as_uint(xi1);
          B.rdy[2][pos] = __float_as_uint(xi2);
          B.rdy[3][pos] = __float_as_uint(s0);
          B.rdy[4][pos] = __float_as_uint(s1);
          B.rdy[5][pos] = __float_as_uint(s2);
          B.rdy[6][pos] = (unsigned)i0;
          B.rdy[7][pos] = (unsigned)i1;
          B.rdy[8][pos] = (unsigned)i2;
          B.rdy[9][pos] = __float_as_uint(D);
          B.rdy[10][pos] = __float_as_uint(eD);
          B.rdy[11][pos] = pid;
          B.rdy[12][pos] = id;
          B.rdy[13][pos] = (unsigned)q;
          B.rdy[14][pos] = (unsigned)pair;
          B.rdy[15][pos] = (unsigned)__double2loint(w);
          B.rdy[16][pos] = (unsigned)__double2hiint(w);
        }
        nwait = 32 - __popc(dead);
        const unsigned take = min(32u, rend - rbeg);
        alive = (unsigned)lane < take;
        if (alive) {
          pid = rbeg + lane;
          Group G = A.groups[gi];
          if ((long long)pid < G.first_particle || (long long)pid >= G.first_particle + (long long)G.n_emitters * G.per_emitter) {
            gi = find_group(A.groups, A.n_groups, (long long)pid);
            G = A.groups[gi];
          }
          // q-major: the lanes of a warp start in different cells
          const unsigned local = pid - (unsigned)G.first_particle;
          q = (int)udiv(local, (unsigned)G.n_emitters, S.group_mag[gi]);
          int e = (int)(local - (unsigned)q * (unsigned)G.n_emitters);
          if (G.perm_off >= 0) e = A.perm[G.perm_off + e];
          band = G.band;
          if (G.kind == 0) {
            w = A.wemit[bc_off + (long long)band * ncells + e];  // from the pass before the trace
          } else {
            w = A.wcoef[((long long)k * A.nb + band) * 6 + G.kind - 1] *
                A.wallTf[in.bface_off + in.wface_off[G.kind - 1] + e];
          }
          alive = (__double_as_longlong(w) << 1) != 0;  // +-0: nothing to trace
          if (alive) {
            int c[3];
            float xi[3], s[3];
            emitter_cell<3>(in, S, k, G.kind, e, c, id);
            st.init(A.seed, inst_id, (uint32_t)band, A.epoch, id, (uint32_t)q);
            emit_segment<3>(st, G.kind, xi, s);
            xi0 = xi[0], xi1 = xi[1], xi2 = xi[2];
            s0 = s[0], s1 = s[1], s2 = s[2];
            g0 = s0 * ih0, g1 = s1 * ih1, g2 = s2 * ih2;
            i0 = c[0], i1 = c[1], i2 = c[2];
            cnt.v[CNT_FLIGHTS] += 1;
          }
        }
        rbeg += take;
        bcbase = bc_off + (long long)band * ncells;
        all_real = A.all_real[(long long)k * A.nb + band] != 0;
        vtm = A.vtm32[(long long)k * A.nb + band];
        if (alive) {
          // the first candidate: its path word from block 0's unused bits, its acceptance word
          // only where some cell of the band may reject
          ub = all_real ? 0u : st.even_word();
          pair = (int)((st.j + 2) >> 1);
          D = __fmul_rn(-__logf(word_uniform<float>(st.first)), vtm);
          eD = fmaf(D, TIE_LOG_REL, vtm * TIE_LOG_ABS);
          kc = 0;
        }
      } else {
        // ---- idle lanes take waiting particles ----
        if (nwait > 0 && (__popc(dead) >= refill || exhausted)) {
          __syncwarp();
          const int rank = __popc(dead & lt_mask);
          if (!alive && rank < nwait) {
            const int pos = nwait - 1 - rank;
            xi0 = __uint_as_float(B.rdy[0][pos]);
            xi1 = __uint_as_float(B.rdy[1][pos]);
            xi2 = __uint_as_float(B.rdy[2][pos]);
            s0 = __uint_as_float(B.rdy[3][pos]);
            s1 = __uint_as_float(B.rdy[4][pos]);
            s2 = __uint_as_float(B.rdy[5][pos]);
            g0 = s0 * ih0, g1 = s1 * ih1, g2 = s2 * ih2;
            i0 = (int)B.rdy[6][pos];
            i1 = (int)B.rdy[7][pos];
            i2 = (int)B.rdy[8][pos];
            D = __uint_as_float(B.rdy[9][pos]);
            eD = __uint_as_float(B.rdy[10][pos]);
            pid = B.rdy[11][pos];
            id = B.rdy[12][pos];
            q = (int)B.rdy[13][pos];
            pair = (int)B.rdy[14][pos];
            kc = pair - (id < (unsigned)ncells ? thermal_uniforms(3) / 2 : wall_uniforms(3) / 2);
            w = __hiloint2double((int)B.rdy[16][pos], (int)B.rdy[15][pos]);
            band = A.nb == 1 ? 0 : A.groups[find_group(A.groups, A.n_groups, (long long)pid)].band;
            vtm = A.vtm32[(long long)k * A.nb + band];
            alive = true;
          }
          nwait = max(0, nwait - __popc(dead));
          __syncwarp();
        }
        // ---- walk: a block of draws, its two candidates (or the second); a particle whose every
        // candidate is real has not got here ----
        bcbase = bc_off + (long long)band * ncells;
        if (alive) {
          st.init_lazy(A.seed, inst_id, (uint32_t)band, A.epoch, id, (uint32_t)q);
          st.load_block((unsigned)pair >> 1);
          second = !(pair & 1);
          const uint32_t uw = second ? st.buf.x : st.buf.z;
          ub = second ? st.buf.y : st.buf.w;
          ++pair;
          const float ell = __fmul_rn(-__logf(word_uniform<float>(uw)), vtm);
          D = __fadd_rn(D, ell);
          eD = fmaf(D, TIE_SUM, fmaf(ell, TIE_LOG_REL, eD + vtm * TIE_LOG_ABS));
        }
      }
      if (alive) {
        // both candidates of a block are looked up before the first is decided (nine in ten of a
        // chain are null): one L2 round trip for two
        const float* ratio = A.ratio32 + bcbase;
        int cell, cell2 = 0, spot2 = SPOT_OUT;
        float ra, ra2 = 0.f, D2 = 0.f, eD2 = 0.f;
        int spot = classify(D, eD, ratio, all_real, cell, ra);
        if (second) {
          const float ell = __fmul_rn(-__logf(word_uniform<float>(st.buf.z)), vtm);
          D2 = __fadd_rn(D, ell);
          eD2 = fmaf(D2, TIE_SUM, fmaf(ell, TIE_LOG_REL, eD + vtm * TIE_LOG_ABS));
          spot2 = classify(D2, eD2, ratio, false, cell2, ra2);
        }
#pragma unroll 1
        for (;;) {
          res = candidate(spot, cell, ra, ub, bcbase, all_real);
          if (res != 0 || !second) break;
          second = false;
          ub = st.buf.w;
          ++pair;
          D = D2;
          eD = eD2;
          spot = spot2;
          cell = cell2;
          ra = ra2;
        }
      }
      close_lane(res);
    }
  }
  flush_lcounts(cnt, A.counters);
}

constexpr size_t CHAIN_SMEM = sizeof(ChainLists) * (CHAIN_NT / 32);

cudaError_t configure_chain(const Ctx* c) {
  const cudaError_t e = allow_shared((const void*)sweep_chain_kernel<false>, c->smem_optin);
  return e != cudaSuccess ? e : allow_shared((const void*)sweep_chain_kernel<true>, c->smem_optin);
}

cudaError_t launch_chain(const Ctx* c, const SweepArgs& a, const StagedArgs& S, bool k32, cudaStream_t s) {
  if (k32) sweep_chain_kernel<true><<<c->sm_count, CHAIN_NT, CHAIN_SMEM, s>>>(a, S);
  else sweep_chain_kernel<false><<<c->sm_count, CHAIN_NT, CHAIN_SMEM, s>>>(a, S);
  return cudaGetLastError();
}

}  // namespace iugkp
