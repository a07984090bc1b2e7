// Internal host/device descriptors of the pplbm library (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>  // header-only: ranges cost nothing unless a profiler is attached
#include <stdint.h>

#include <vector>

#include "pplbm.h"

namespace pplbm {

// An NVTX range around a host call (step, chunk, readback), named for the profiler's timeline.
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

// Per-tile partial sums folded by the last CTA of an instance:
// mass, energy, T summed over the heater-adjacent row, inlet flux, outlet flux.
constexpr int NPART = 9;  // mass, energy, heater row T, inflow, outflow, vapour area, wall / heater / zone vapour
// The tiles of a launch add their partial sums into NPART signed 64-bit fixed-point totals;
// total j has 52 - ceil(log2(m_j)) fraction bits, m_j the most nodes that feed it (nx ny for
// mass, energy and the vapour counts, nx for the heater row, ny for the inlet and outlet
// columns).  Every per-node term is at most 1024 in magnitude, so a total stays below 2^62,
// and integer addition is exact and commutative, so the totals do not depend on the order in
// which tiles finish.
constexpr int FIX_BITS = 52;
constexpr int NDIAG = 12;  // LBM_D_COUNT
constexpr int RING = 1024;  // diagnostics records kept per instance

enum : int { GEOM_PERIODIC = 0, GEOM_CHANNEL = 1, GEOM_WALLS = 2, GEOM_POOL = 3 };
enum : int { MODE_STEP = 0, MODE_FIELDS = 1, MODE_POPS = 2, MODE_MOMENTS = 3 };
enum : unsigned { STATUS_UNSTABLE = 1u, STATUS_TIMEOUT = 2u, STATUS_BOUNDS = 4u };

// Device-resident mutable state of one lattice instance.
// Step n uses the slots n & 1 of counter and p_probe and the slot n % 4 of the open-end mass
// exchange: the overlapped persistent loop has tiles of two consecutive steps in flight.
struct InstState {
  long long step;       // steps completed
  int local_read;       // 1: buffer (step & 1) holds post-stream populations (after init/load)
  unsigned int status;  // sticky STATUS_* bits, cleared by the host
  unsigned int counter[2];   // tiles of step n that have posted their partials, in slot n & 1
  unsigned int bounds_hits;  // accesses a bounds-checked build rejected (STATUS_BOUNDS), else 0
  unsigned int open_posted[4];  // open-end tiles of step n that posted open_mass, in slot n % 4
  int pad0;
  double rho_avg[2];    // domain-mean rho of step n in slot n & 1 (buoyancy of step n+1, Eq. 14)
  double p_probe[4];    // EOS pressure at (1, ny/2) and (nx-2, ny/2) of step n in slots 2 (n & 1) + {0, 1}
  long long open_mass[4];  // fixed-point mass that step n's pull took in and let out through the
                           // open ends (created minus lost populations), in slot n % 4
};

// D2Q9 weights.  In FP32 the rounded 4/9, 1/9, 1/36 sum to 1 + 7.6e-9, which would
// create mass (and energy) in every collision in proportion to the stored deviation;
// the FP32 set below (1/36 lowered by one ulp) sums to exactly 1.
template <typename Real>
struct LatWeights {
  __host__ __device__ static constexpr Real w0() { return Real(4.0 / 9.0); }
  __host__ __device__ static constexpr Real w1() { return Real(1.0 / 9.0); }
  __host__ __device__ static constexpr Real w5() { return Real(1.0 / 36.0); }
};
template <>
struct LatWeights<float> {
  __host__ __device__ static constexpr float w0() { return 0x1.c71c72p-2f; }
  __host__ __device__ static constexpr float w1() { return 0x1.c71c72p-4f; }
  __host__ __device__ static constexpr float w5() { return 0x1.c71c70p-6f; }
};
// ---------------------------------------------------------------------------
// Per-instance constants of the update, converted once per CTA to the compute
// precision (the instance descriptor holds them in FP64).
// ---------------------------------------------------------------------------
template <typename Real>
struct KConst {
  Real omega_f, omega_g, a, b, R, kappa, inv_sqrtTc, psi_scale, beta, G2, Gh, mix, g_a, inv_cv;
  Real T0, rho_ref, T_ref, alpha0, u_in, drho_out, dT_in, dT_heat;
  // FP32 pseudopotential reference state (zero in FP64)
  Real inv_u1r, inv_Dr, sqrtT_r, sa_r, rr2_Dr, rad_ref, psi_ref, p_ref;
  // force on a row next to the bottom wall: wall0 + d * wall1 (the top wall: minus that)
  Real wall0, wall1;
  Real rho_ref_minus_avg;  // rho_ref - rho_avg of the previous step (buoyancy, Eq. 14)
  Real drho_vapor;         // rho_vapor - rho_ref: vapour when drho < drho_vapor
  // products of the constants above, formed once (host doubles): R / (1 - b rho_ref),
  // a / D(rho_ref), 2 b rho_ref, -kappa / sqrt(Tc), a rho_ref^2 / D(rho_ref)
  Real R_u1r, a_Dr, twob_rr, nk_sTc, a_rr2_Dr;
  // FP64 step: G / 4, 1 + kappa, psi_scale R, psi_scale a, psi_scale / 3, R / c_v, -a kappa / (sqrt(Tc) c_v)
  Real Ghh, kappa1, R_ps, a_ps, ps_3, R_cv, ank_cv;
};

// Constants of the packed step, each held twice so that a packed instruction takes it as one
// 64-bit operand; products are formed on the host in FP64.
struct KPair {
  float2 rho_ref, T_ref;
  float2 b;  // Eq. 12
  // with s = sqrt(alpha / alpha(T_ref)) = 1 + m1 (sqrt T - sqrt T_ref), D = 1 + 2 b rho - (b rho)^2:
  // psi^2 - psi_ref^2 = cA (drho T / (1 - b rho) + rho_ref dT) + cB s^2 drho (s3 rho + rho_ref) / D
  //                     + cK (s - 1) / m1 (s + 1) + c3 drho   (Eqs. 11, 12)
  float2 m1, cA, cB, cK, c3, s3, T0;
  float2 sqrtT_r, rad_ref, psi_ref;
  float2 cR, cS;            // T (dp/dT)_rho / (rho c_v) = T (cR / (1 - b rho) + cS s / sqrt T rho / D)
  float2 G2, Gh, Ghh;       // 2 G, G / 2, G / 4
  float2 nbeta, npsi_ref, nmix;  // Eq. 8: -beta, -psi_ref, -(1 - beta) / 2
  float2 ng_a, wall0, wall1;
  float2 omega_f, keep_f, omega_g, keep_g;
  float inv_ps, p_ref;              // probes only: dp = drad / psi_scale + drho / 3
};

// The converted constants of the FP32 strip step.
struct StripConst {
  KConst<float> C;
  KPair P;
};

// Read-only description of one lattice instance (host-filled, device-resident).
struct Inst {
  int nx, ny, pitch, geometry;
  long long plane;      // elements per population plane (pitch * ny)
  void* f[2];           // population double buffer: 9 planes each (storage precision)
  void* g[2];
  int multiphase, pad1;
  double omega_f, omega_g;          // 1/tau_f, 1/tau_g
  double a, b, R, kappa, sqrtTc, inv_sqrtTc;
  double psi_scale;                 // 2/(c0 G) of Eq. 11
  double beta, G2, Ghalf;           // Eq. 8 beta; Eq. 10 g1 = 2G, g2 = G/2
  double Gwet_psiw;                 // G_wet * psi(rho_w, T0) of Eq. 15
  double g_a, inv_cv;
  double T0, T_in, T_heat, u_in, rho_out;
  double rho_ref, T_ref;            // storage offsets: f stored as f - w_i rho_ref, g as g - w_i T_ref
  double alpha0;                    // alpha(T0) of Eq. 12 for isothermal runs
  // FP32 reference state of the pseudopotential: psi is carried as psi - psi_ref,
  // evaluated from exact difference forms of Eq. 12 in rho - rho_ref and T - T_ref
  double psi_ref, rad_ref, p_ref, inv_u1r, inv_Dr, sa_r, sqrtT_r, rr2_Dr;
  int heater_x0, heater_len;
  long long heat_on_step;
  double rho_vapor;                 // vapour threshold of the bubble diagnostics
  int source_model, bubble_stats;   // 0 Gong-Cheng, 1 Hazi-Markus (first Eq. 19); count vapour nodes
  void* rho_prev;                   // rho^(n-1) - rho_ref per node (storage precision, pitch layout)
  const void* tmaps;                // FP32: 4 tensor maps of 128 bytes (f of buffers 0, 1, then g); or null
  InstState* st;
  unsigned long long* sums;         // NPART fixed-point totals of the current launch (zero between launches)
  double fix_scale[NPART];          // 2^f_j, f_j the fraction bits of total j
  double fix_unscale[NPART];        // 2^-f_j
  double* ring;                     // RING records of NDIAG doubles
  // Element offsets within a population buffer: population i of node n sits at n + poff[i]
  // (poff[i] = i * plane), and on a node with no wall or open-end link it is pulled from
  // n + loff[i] (the node n - c_i, in plane i: loff[i] = poff[i] - c_iy pitch - c_ix).
  int loff[9], poff[9];
  // Derived constants of the step, formed on the host only (so that every kernel converts the
  // same doubles): (1 - beta)/2 of Eq. 8; the outlet density, inlet and heater temperatures as
  // deviations from the storage references; the vapour threshold as a density deviation; and
  // the reference parts of Eqs. 9 and 15 on a row next to the bottom wall, wall0 + d wall1 with
  // d = psi - psi_ref (its fluid neighbours have sum G_i c_iy = 3G and its solid neighbours
  // sum w_i c_iy = -1/6; the two parts cancel exactly for a balanced wall, which keeps the FP32
  // force free of the cancellation).
  double mix, drho_out, dT_in, dT_heat, drho_vapor, wall0, wall1;
  // products of constants of the FP32 equation of state, formed on the host: R / (1 - b rho_ref),
  // a / D(rho_ref) with D(rho) = 1 + 2 b rho - (b rho)^2, 2 b rho_ref, -kappa / sqrt(Tc),
  // a rho_ref^2 / D(rho_ref)
  double R_u1r, a_Dr, twob_rr, nk_sTc, a_rr2_Dr;
  StripConst strip;  // FP32; last: the one-column kernels copy what comes before it
};

// Every member is a conversion of a descriptor value (derived values are formed once, on the
// host, in fill_inst), so the host's copy (kernel parameter) and a CTA's copy (shared memory)
// are bit-identical.
template <typename Real>
__host__ __device__ inline void fill_consts(KConst<Real>& c, const Inst& I, double rho_avg_prev) {
  c.omega_f = Real(I.omega_f);
  c.omega_g = Real(I.omega_g);
  c.a = Real(I.a);
  c.b = Real(I.b);
  c.R = Real(I.R);
  c.kappa = Real(I.kappa);
  c.inv_sqrtTc = Real(I.inv_sqrtTc);
  c.psi_scale = Real(I.psi_scale);
  c.beta = Real(I.beta);
  c.G2 = Real(I.G2);
  c.Gh = Real(I.Ghalf);
  c.mix = Real(I.mix);
  c.g_a = Real(I.g_a);
  c.inv_cv = Real(I.inv_cv);
  c.T0 = Real(I.T0);
  c.rho_ref = Real(I.rho_ref);
  c.T_ref = Real(I.T_ref);
  c.alpha0 = Real(I.alpha0);
  c.u_in = Real(I.u_in);
  c.drho_out = Real(I.drho_out);
  c.dT_in = Real(I.dT_in);
  c.dT_heat = Real(I.dT_heat);
  c.inv_u1r = Real(I.inv_u1r);
  c.inv_Dr = Real(I.inv_Dr);
  c.sqrtT_r = Real(I.sqrtT_r);
  c.sa_r = Real(I.sa_r);
  c.rr2_Dr = Real(I.rr2_Dr);
  c.rad_ref = Real(I.rad_ref);
  c.psi_ref = Real(I.psi_ref);
  c.p_ref = Real(I.p_ref);
  c.wall0 = Real(I.wall0);
  c.wall1 = Real(I.wall1);
  c.rho_ref_minus_avg = Real(I.rho_ref - rho_avg_prev);
  c.drho_vapor = Real(I.drho_vapor);
  c.R_u1r = Real(I.R_u1r);
  c.a_Dr = Real(I.a_Dr);
  c.twob_rr = Real(I.twob_rr);
  c.nk_sTc = Real(I.nk_sTc);
  c.a_rr2_Dr = Real(I.a_rr2_Dr);
  c.Ghh = Real(0.5 * I.Ghalf);
  c.kappa1 = Real(1.0 + I.kappa);
  c.R_ps = Real(I.R * I.psi_scale);
  c.a_ps = Real(I.a * I.psi_scale);
  c.ps_3 = Real(I.psi_scale * (1.0 / 3.0));
  c.R_cv = Real(I.R * I.inv_cv);
  c.ank_cv = Real(I.a * I.nk_sTc * I.inv_cv);
}

__host__ __device__ inline float2 pair_of(double v) { return make_float2((float)v, (float)v); }

__host__ __device__ inline void fill_pair_consts(KPair& P, const Inst& I) {
  const double ps = I.psi_scale, sr = I.sa_r;
  P.rho_ref = pair_of(I.rho_ref);
  P.T_ref = pair_of(I.T_ref);
  P.b = pair_of(I.b);
  P.m1 = pair_of(sr != 0.0 ? I.nk_sTc / sr : 0.0);
  P.cA = pair_of(I.R_u1r * ps);
  P.cB = pair_of(-I.a_Dr * sr * sr * ps);
  P.cK = pair_of(-I.a_rr2_Dr * I.nk_sTc * sr * ps);
  P.c3 = pair_of(-ps / 3.0);
  P.s3 = pair_of(1.0 + I.twob_rr);
  P.T0 = pair_of(I.T0);
  P.sqrtT_r = pair_of(I.sqrtT_r);
  P.rad_ref = pair_of(I.rad_ref);
  P.psi_ref = pair_of(I.psi_ref);
  P.cR = pair_of(I.R * I.inv_cv);
  P.cS = pair_of(-I.a * I.nk_sTc * sr * I.inv_cv);
  P.G2 = pair_of(I.G2);
  P.Gh = pair_of(I.Ghalf);
  P.Ghh = pair_of(0.5 * I.Ghalf);
  P.nbeta = pair_of(-I.beta);
  P.npsi_ref = pair_of(-I.psi_ref);
  P.nmix = pair_of(-I.mix);
  P.ng_a = pair_of(-I.g_a);
  P.wall0 = pair_of(I.wall0);
  P.wall1 = pair_of(I.wall1);
  P.omega_f = pair_of(I.omega_f);
  // 1 - omega of the FP32 omega, exactly: a collision must not create mass or energy
  P.keep_f = make_float2(1.0f - P.omega_f.x, 1.0f - P.omega_f.x);
  P.omega_g = pair_of(I.omega_g);
  P.keep_g = make_float2(1.0f - P.omega_g.x, 1.0f - P.omega_g.x);
  P.inv_ps = ps != 0.0 ? (float)(1.0 / ps) : 0.0f;
  P.p_ref = (float)I.p_ref;
}

// State of the grid-wide barrier between the steps of a persistent launch (device memory,
// zeroed by the host before every persistent launch).  count: CTAs arrived at the current
// barrier; gen: barriers completed; status: 1 once a CTA gave up waiting; next[2]: the
// dynamic tile counters of even and odd steps.
//
// Overlapped form (FlowPlan.enabled, a parameter of the launch; a lattice or a batch whose
// tiling has more tiles than resident CTAs): the CTAs draw (step, tile) tickets in order from
// `claim`, and a tile of step s waits only for what it reads, instead of a barrier for all the
// tiles: the tiles of its instance around it to have finished step s - 1 (cell_done), step
// s - 2 of its instance to be complete (its mean density), and the instance's open-end tiles
// of step s - 1 to have posted the mass that crossed the inlet and outlet; its buoyancy mean is
// the mean of step s - 2 plus that mass over the nodes (Eq. 14).  Tiles of two consecutive
// steps run at once, so the end of one step overlaps the start of the next.
struct FlowInst {  // one instance's tiling
  int strips, nbands, tile_w;             // tiles per band, bands per step, output columns per tile
  int tall_rows, tall_count, short_rows;  // band layout (row y -> band)
  int n_open;                             // tiles per step with an open end
  int perx, pery;                         // strips wrap in x (walls, periodic), bands in y (periodic)
  int pad;
  long long cell_base;                    // the instance's first tile position in cell_done
};
struct FlowPlan {
  int enabled;
  int ninst;
  FlowInst single;                 // the instance of a single-lattice launch (inst == nullptr)
  const FlowInst* inst;            // a batch's table (device memory), indexed by Tile.inst
  long long* step0;                // per instance: its step when the launch starts (written by the
                                   // launch's first CTA before the tickets start)
  unsigned long long* cell_done;   // per tile position (cell_base + band * strips + strip): steps
                                   // of this launch it has finished (zeroed before the launch)
};
// Flat persistent launch (lbm_flat.cuh): a CTA per tile, a warp per row, every CTA owning its
// tiles for all the steps.  A tile of step s waits for the tiles around it (deps: what its pulls
// read) to have finished step s - 1, and for the mass totals of step s - 1 to be complete.
constexpr int FLAT_MAX_DEPS = 25;
// Output columns of a strip of at most w (even) columns with `left` columns of the lattice from its
// first on: what is left, rounded up to a lane's two.  The lanes past the last column of a lattice
// that wraps then pull no column beyond those that the tile waits for.
__host__ __device__ inline int strip_columns(int w, int left) { return left < w ? (left + 1) / 2 * 2 : w; }
struct FlatTile {
  short inst, wout;            // output columns [x0, x0 + wout), rows [y0, y0 + rows)
  int x0, y0, rows;
  int ntiles;                  // tiles of the instance
  int ndeps;
  int deps[FLAT_MAX_DEPS];     // positions in the launch's tile table
  unsigned char dep_rows[FLAT_MAX_DEPS + 3];  // rows of those tiles: each adds one count per row and step
};
// Per instance, zeroed before the launch: step s uses slot s % 4 of the totals, of the pressure
// probes and of the counts of tiles; the last tile of step s clears the slot of step s - 1, which
// every tile has read by then.  What different warps poll and add to lies on different cache lines.
struct __align__(128) FlatSlot {
  unsigned int count;                           // tiles that have added their mass
  unsigned int pad0[31];
  unsigned long long sums[16];                  // NPART totals, the mass first
  unsigned int complete;                        // tiles that have added all their sums
  unsigned int pad1[31];
  double probe[16];
};
struct FlatState {
  FlatSlot slot[4];
};
constexpr int FLAT_DONE_STRIDE = 32;  // a tile's count of finished rows, one per cache line
struct GridBar {
  unsigned int count, gen, status, pad;
  unsigned int next[2];
  unsigned long long claim;  // overlapped form: (step, tile) tickets drawn in this launch
};
// Bounded waits of the persistent launch: a CTA stops waiting at a barrier after wait_ns
// nanoseconds of polling, or after max_polls polls when max_polls > 0 (a test lowers it to
// make the wait run out while the other CTAs are still busy).
constexpr unsigned long long BARRIER_WAIT_NS = 5000000000ull;

// One CTA's work: output columns [x0, x0 + W) of instance `inst`, rows [y0, y1).
struct Tile {
  int inst, x0, y0, y1;
  int local;   // index of this tile among its instance's tiles (partials slot)
  int ntiles;  // tiles of this instance in the launch
  int interior;  // 1: every column the tile pulls, [x0 - 2, x0 + cols - 6), lies in [1, nx - 2] of a
                 // channel or walls lattice (no open end, no wrap): the interior path may take it
  int open_end;  // 1: the tile's output columns include the inlet or the outlet of a channel
};
// Whether a tile of a cols-thread step tiling starting at column x0 may take the interior path.
inline int tile_is_interior(int geometry, int nx, int cols, int x0) {
  return (geometry == GEOM_CHANNEL || geometry == GEOM_WALLS) && x0 - 2 >= 1 && x0 + (cols - 8) + 1 <= nx - 2;
}
// Tiles that take the general loop (dispatched before the interior tiles of their class).
inline bool general_tile(const Tile& t) { return !t.interior; }

// Launchers (defined per precision).  Tiles must have been built for `cols`.
// kernel: a resolved form (resolve_kernel): LBM_KERNEL_SCALAR, _INTERIOR, _TMA or FORM_STRIP.
// flags: STEP_FULL, the instances use the pool geometry, the Hazi-Markus source or bubble
// statistics, which only the step's full form handles (the lean form leaves them out of the hot
// loop); STEP_RELAX, tau_f != 1 (the strip kernel then keeps the pulled f for the collision).
// h_inst: host copy of the launch's only instance (the lean scalar step then takes its
// constants as a kernel parameter), or null for launches over several instances.
// max_polls: poll cap of the TMA form's row waits (0: its full limit; lbm_set_wait_limit).
cudaError_t launch_lbm(int fp64, int thermal, int cols, int mode, int kernel, int flags, const Inst* d_inst,
                       const Tile* d_tiles, int ntiles, cudaStream_t s, const Inst* h_inst = nullptr,
                       unsigned max_polls = 0);
// nsteps steps of the flat FP32 kernel in one cooperative launch of `grid` CTAs of `warps` warps over
// the tiles of build_flat_tiles (tile i on CTA i % grid); fstate (per instance) and done (per
// tile) zeroed.
cudaError_t launch_flat(int thermal, int flags, int warps, const Inst* d_inst, const FlatTile* d_tiles, int ntiles,
                        int grid, int nsteps, FlatState* fstate, unsigned* done, GridBar* bar, unsigned max_polls,
                        cudaStream_t s, const Inst* h_inst);
int flat_resident_ctas(int thermal, int flags, bool single, int warps);
struct FlatSize {
  int nx, ny;
};
bool build_flat_tiles(int inst, int nx, int ny, int geometry, int rows, std::vector<FlatTile>& out);
// per_sm_by_warps: resident CTAs per SM by warps per CTA (indices 0 .. 20).
int flat_rows(const std::vector<FlatSize>& sizes, int sms, int max_rounds, const int* per_sm_by_warps);
// The most tiles that a lattice's flat launch takes on `sms` SMs with at most max_rounds tiles a CTA; 0
// where it is too large for it at every tile height.
int flat_max_tiles(int nx, int ny, int sms, int max_rounds);
constexpr int FLAT_MAX_STEPS = 1 << 27;  // of a launch: steps times rows stay below 2^32
constexpr double FLAT_ROUND_COST = 10.0;  // in warps
// Rounds (tiles per CTA) up to which the flat launch is taken.  A round costs about 6 us whatever the
// size, the strip kernel no less than 18 us a step: 1500 x 150 (2 rounds) 13.1 us against 21.2 (the
// best of five strip tilings and loops), 1800 x 160 (3) 18.2 against 21.2; with the limit raised, 2000
// x 200 (4) 24.2 against 24.6, 2500 x 220 (5) 31.3 against 26.7.  A batch's strip kernel reads its
// constants from shared memory and is a little slower: three 128 x 512 pools 19.0 against 26.6 us,
// four 21.3 against 29.1, five (4 rounds) 27.8 against 30.9, six (5) 34.1 against 31.8.
constexpr int FLAT_AUTO_ROUNDS = 3, FLAT_BATCH_ROUNDS = 4;
// nsteps steps of the step kernel in one cooperative launch (tiles drawn dynamically from a
// counter, a bounded grid barrier between steps; MODE_STEP only).  grid <= resident CTAs of
// the device; bar: zeroed GridBar in device memory.
// flow.enabled: the overlapped form (one instance; more tiles than resident CTAs).
cudaError_t launch_persistent(int fp64, int thermal, int cols, int kernel, int flags, const Inst* d_inst,
                              const Tile* d_tiles, int ntiles, int nsteps, GridBar* bar, unsigned max_polls,
                              cudaStream_t s, const Inst* h_inst, const FlowPlan& flow);
// CTAs one persistent launch may hold on the current device (SMs x resident CTAs per SM).
long long persistent_slots(int fp64, int thermal, int cols, int kernel, int flags, bool single);
// Whether an instance needs the step's full form.
inline bool needs_full_step(const Inst& I) {
  return I.geometry == GEOM_POOL || I.source_model != 0 || I.bubble_stats != 0;
}
enum : int { STEP_FULL = 1, STEP_RELAX = 2 };
inline int step_flags(const Inst& I) {
  return (needs_full_step(I) ? STEP_FULL : 0) | (I.omega_f != 1.0 ? STEP_RELAX : 0);
}
// The kernel a launch takes for a requested LBM_KERNEL_* value.  In FP32, LBM_KERNEL_AUTO,
// _INTERIOR and _PAIRED all take the strip kernel (lbm_strip.cuh), which handles every option and
// is the fastest on GB300.  In FP64, LBM_KERNEL_AUTO and _INTERIOR take the one-column kernel
// with its interior path (tiles away from open ends and wraps run a loop without any per-node
// boundary logic; the others run the general loop) whenever the step's lean form applies, else
// the plain one-column kernel.  The TMA kernel needs FP32, 128-column tiles, the step's lean form
// and the instances' tensor maps (tmaps: all instances of the launch have them).
constexpr int TMA_TILE_COLS = 128;
constexpr int FORM_STRIP = 16;  // beside the LBM_KERNEL_* values
inline int resolve_kernel(int requested, int fp64, bool full, bool tmaps, int cols) {
  if (requested == LBM_KERNEL_AUTO || requested == LBM_KERNEL_INTERIOR)
    return !fp64 ? FORM_STRIP : full ? LBM_KERNEL_SCALAR : LBM_KERNEL_INTERIOR;
  if (fp64) return LBM_KERNEL_SCALAR;
  if (requested == LBM_KERNEL_PAIRED) return FORM_STRIP;
  if (requested == LBM_KERNEL_TMA && !full && tmaps && cols == TMA_TILE_COLS) return LBM_KERNEL_TMA;
  return LBM_KERNEL_SCALAR;
}
// The LBM_KERNEL_* value reported for it: the strip kernel goes by the form that was asked for,
// "scalar" where that form's boundary logic is the per-node one (the full form, Hazi-Markus).
inline int reported_kernel(int requested, int form, bool full, bool hazi) {
  if (form != FORM_STRIP) return form;
  if (requested == LBM_KERNEL_PAIRED) return hazi ? LBM_KERNEL_SCALAR : LBM_KERNEL_PAIRED;
  return full ? LBM_KERNEL_SCALAR : LBM_KERNEL_INTERIOR;
}
// The LBM_FORM_* value of the kernel that runs.
inline int executed_form(int form, bool flat) {
  if (flat) return LBM_FORM_FLAT;
  return form == FORM_STRIP ? LBM_FORM_STRIP : form == LBM_KERNEL_TMA ? LBM_FORM_TMA
         : form == LBM_KERNEL_INTERIOR ? LBM_FORM_INTERIOR : LBM_FORM_SCALAR;
}
// Whether a kernel has a persistent form.
inline bool has_persistent(int form) {
  return form == LBM_KERNEL_SCALAR || form == LBM_KERNEL_INTERIOR || form == FORM_STRIP;
}
// f = f^eq(rho,u), g = g^eq(T,u) into buffer 0 from 4 planes of nx*ny doubles (rho, ux, uy, T).
cudaError_t launch_init_from_fields(int fp64, const Inst* d_inst, int nx, int ny, const double* d_fields,
                                    int has_T, cudaStream_t s);
// Built-in initial state (uniform or seeded disk) into buffer 0.
struct InitSpec {
  int kind;
  double rho_in, rho_out, radius, width, amp, T0;
  unsigned long long seed;
  int instance;
};
cudaError_t launch_init_builtin(int fp64, const Inst* d_inst, int nx, int ny, InitSpec spec, cudaStream_t s);

bool cols_supported(int cols);

// Host helpers shared by the context API and the allocation-free step.
// check_params: nullptr when p is valid for an nx x ny lattice, else the reason.
const char* check_params(int nx, int ny, const lbm_params* p);
// fill_inst: the physics part of an instance descriptor (buffer and scratch pointers
// are left null); nullptr on success, else the reason.
const char* fill_inst(Inst& I, const lbm_params* p, int nx, int ny, int pitch, long long plane, int fp64);
// Rows per band of the default tiling for CTAs of `cols` threads.
// Rows per band of a cols-wide step tiling of an nx x ny lattice: the band height
// that covers the lattice in the fewest row-iterations per CTA slot, counting the 4
// halo rows (plus about one row of fixed cost) every band adds, the `slots` CTAs one
// wave holds and half a tile of tail.  Never below 4 rows unless the lattice is lower.
int default_band_rows(int nx, int ny, int cols, long long slots);
// Rows of a step tiling, per strip of cols - 8 columns: tall_count bands of tall_rows from the
// bottom, then bands of short_rows (the last one possibly lower) up to the top; every strip's
// tall bands are dispatched before any short band (uniform tilings: tall_count = 0).
struct BandPlan {
  int tall_rows, tall_count, short_rows;
};
// The default step tiling of an nx x ny lattice for `slots` CTA slots: the uniform band height
// of default_band_rows, or, where the same cost model finds it cheaper, tall bands of 2h rows
// followed by about one wave of short bands of h rows, which the block scheduler dispatches
// last, so the end of the step is filled by short tiles while most rows pay the halo of tall
// bands only.
BandPlan default_band_plan(int nx, int ny, int cols, long long slots);
// CTAs of the step kernel (storage precision, thermal flag, tile columns, kernel
// form) that one wave of the current device holds: SMs x resident CTAs per SM.
long long step_wave_slots(int fp64, int thermal, int cols, int kernel, int flags = 0);
int resident_ctas_f32(int thermal, int cols, int kernel, int flags);
int resident_ctas_f64(int thermal, int cols, int kernel);
// The instance descriptor of a context (device pointers included), for batching.
Inst lbm_internal_inst(const lbm_ctx* c);
// Changes whenever the context's descriptor is rewritten (parameters or a loaded state).
unsigned long long lbm_internal_params_gen(const lbm_ctx* c);
// A context for a batch's member: as lbm_create, without a flat launch of its own.
lbm_status lbm_internal_create_member(lbm_ctx** out, int32_t nx, int32_t ny, lbm_precision prec, int32_t device,
                                      void* stream);

}  // namespace pplbm
