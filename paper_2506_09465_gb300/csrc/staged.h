// Work distribution of the staged sweep (sweep_staged.cu), built on the host.
#pragma once

namespace iugkp {

constexpr int STAGED_NT = 1024;                 // threads per persistent block
constexpr int WALK_MIN_LANES = 8;               // landing chains: fewest lanes worth a step

// 3D sweep (sweep_chain.cu): threads of a block (five warps per scheduler: with four 17.3 ms, five
// 15.4 ms, six 17.7 ms on four boxes up to 64^3), and the idle lanes that trigger a refill (2 to 4:
// the same, 8: 3 % more).
constexpr int CHAIN_NT = 640;
constexpr int CHAIN_REFILL = 4;

// Shared-memory x-face window: one 32-bit word per face holding the low word of a 64-bit
// fixed-point sum in units of w_max 2^-26 (a contribution is below 2^26 units); words start
// at 2^31, and a wrap of the word adds +-2^32 units to the
// face's 64-bit sum at once.
constexpr double WIN_SCALE = 0x1p26;
constexpr unsigned WIN_BIAS = 0x80000000u;

// Copies of the two-group exit tally GX (one per block, by block index modulo the count),
// summed when the untallied faces are derived. Exits through one wall pile onto a few hundred
// faces (a single 128 x 128 instance at Kn 10 sends ~4e6 exits to 256 of them); FP64
// atomics to one address serialise at its L2 slice, so one copy made the sweep's time
// depend on which slices those lines landed in.
constexpr int GX_COPIES = 16;

struct StagedArgs {
  int n_inst;
  unsigned long long* inst_next;  // [n_inst] next unclaimed forward particle of each instance
  const long long* inst_end;      // [n_inst] end of each instance's forward particle range
  const double* cost_prefix;      // [n_inst] prefix sums of the estimated cost
  double cost_total;
  const int2* window;             // [n_inst] {first x-face, count} tallied in shared memory
  const double* wmax;             // [n_inst] largest |particle weight| of the sweep
  int warp_grab;                  // particles a warp claims at a time
  int refill;                     // idle lanes that trigger a refill (0: per-instance default)
  int walk_k;                     // crossings per lane between bulk steps
  // division magics M = floor((2^32 - 1) / d) of the divisors d below
  const unsigned* group_mag;      // [forward groups] d = emitters of the group
  const unsigned* mag_n0;         // [n_inst] d = n_x
  const unsigned* mag_n1;         // [n_inst] d = n_y
  const unsigned* mag_wall;       // [n_inst * 3] d = cells along the first tangential axis of each wall
  // compensated FP32 tallies (IUGKP_TALLY_STAGED_K32): {high word, error word} per entry
  float2* R32;                    // [nb * total_cells]
  float2* W32;                    // [nb * total_cells] or null
  float2* F32;                    // [total_faces] face tallies that miss the window, or null
  // Two-group face tallies (2D instances whose faces all fit the window): a particle whose
  // path per cell along x is at least that along y (d_x >= d_y) is in the x-group and
  // tallies the faces normal to x it crosses; the others (y-group) tally the faces normal
  // to y. The untallied faces of each group follow from that group's own power balance.
  double* DY;                     // [total_cells] y-group: absorbed minus emitted power per cell
  double* EY;                     // [total_bfaces] y-group wall emission per boundary face (signed
                                  // flux: + on the low walls, - on the high walls)
  double* GX;                     // [GX_COPIES][total_bfaces] exits of the x-group through the low
                                  // y-wall and of the y-group through the low x-wall (signed flux)
  long long gx_stride;            // total_bfaces: entries per copy of GX
  long long* Fi;                  // [total_faces] fixed-point face sums in units of the instance's q
  // Particles whose FP32 walk lies within rounding of a decision of the FP64 walk are left
  // untallied and replayed by the FP64 walk after the sweep (replay_kernel): entry
  // {forward index, (candidates already tallied << 1) | y-group}.
  uint2* defer;                   // [defer_cap]
  unsigned* defer_n;              // entries pushed by this sweep (beyond defer_cap: overflow)
  unsigned defer_cap;
  int* err;                       // device error word (ERR_DEFER on overflow)
  // Landing sweeps only (else null): bitmap of the particles beyond the queue, zero between launches
  // (the replay clears what it takes).
  unsigned* over;                 // [over_words]
  unsigned over_words;
#ifdef __CUDACC__
  // this block's copy of GX
  __device__ __forceinline__ double* gx() const {
    return GX + (long long)(blockIdx.x % (unsigned)GX_COPIES) * gx_stride;
  }
#endif
};

// The pass before a trace (closing.cu).
struct PrologueArgs {
  int n_clear;
  unsigned long long* clear[12];  // buffers to clear and their sizes in 8-byte words
  long long words[12];
  int n_inst;
  unsigned long long* next;       // [n_inst] claim counters <- next_from, or null
  const long long* next_from;
  int wmax_blocks;                // blocks of the emitter weights (0: none)
  const int* bpre;                // [groups + 1] first block of each group
  unsigned long long* wpart;      // [wmax_blocks]
  unsigned long long* wmax;       // [n_inst]
  unsigned* ticket;               // 0 between launches
};

// The pass after a 2D staged trace (closing.cu).
struct Close2D {
  const int2* window;
  const double* wmax;
  const long long* Fi;
  const double* Fx;
  const double* bal;              // [cells] balances, or null (one band: formed on the spot)
  const double* Vm;
  const double* wall_unit;
  const double* DY;
  const double* EY;
  const double* GX;
  long long gx_stride;
  unsigned* ticket;               // [n_inst], 0 between launches
  int line_blocks;
};

// Landing sweeps (land.cu).
constexpr int LAND_NT = 256;          // threads per block
constexpr int LAND_QCH = 16;          // particles per emitter and task at most
constexpr int LAND_WARPS_PER_SM = 40; // resident warps the task size is chosen for
constexpr int LAND_REFILL = 8;        // idle lanes that trigger a refill (null-candidate chains)

// Filtered FP64 sweep (exact.cu): copies of the 1D trees over the faces at most, and the faces of all of
// them together (beyond, addresses are seldom the same); the
// candidates after which a particle (there and in a landing sweep with FP64 tracking) goes to the
// replay, which keeps the step budget.
constexpr int EXACT_NODE_COPIES = 16;
constexpr long long EXACT_NODE_FACES = 1 << 15;
constexpr int EXACT_MAX_CANDIDATES = 1 << 20;
constexpr long long EXACT_MIN_BUDGET = 1ll << 24;  // smaller step budgets take the plain kernel

// A group's tasks: tiles of tw emitters (reps particles of an emitter side by side where tw is
// at most 16) x runs of qch * reps particles per emitter, tiles fastest; task0 is its first.
struct LandGroup {
  unsigned first;                 // first particle (forward or adjoint numbering)
  int inst, band, kind, ne, per, perm_off;
  int tw, ntile, reps;
  unsigned task0;
  int next;                       // group of the next band of the same emitters, or -1 (land_tasks)
  int pass0;                      // passes of the bands before this one in such a chain
};

struct LandArgs {
  const LandGroup* groups;
  int n_groups;
  unsigned n_tasks;
  int qch;
  unsigned long long* next;       // next unclaimed task (or particle, where chains are followed)
  const double* lamVm;            // adjoint: [cells] lambda / (V m)
  unsigned max_j;                 // chains: uniforms after which a particle goes to the replay
};

// Tasks of the pass-synchronous 2D sweep: those of an instance are contiguous.
struct SyncArgs {
  LandArgs L;
  const unsigned* task_end;       // [n_inst]
};

}  // namespace iugkp
