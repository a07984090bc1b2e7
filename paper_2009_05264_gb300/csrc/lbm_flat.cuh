// FP32 step for lattices of a few tiles per SM: a CTA per tile, a warp per row, all steps of a call
// in one cooperative launch.
//
// The same row arithmetic as the strip kernel (LaneStep), with the rows of a tile side by side in
// the warps of a CTA instead of one after another in one warp: warp w holds row y0 - 2 + w of the
// tile, its populations pulled straight into registers; the rows exchange psi and u_act through
// shared memory around two barriers (moments and EOS; force and f collision; g collision).
//
// Why: a small lattice's step is a chain of latencies, not of work.  Marching eight rows (four and
// the halo) in one warp costs eight dependent passes of about 600 instructions at six cycles each,
// 16 us of a 21 us step on 1000 x 100; here the chain is one row's, and a tile of up to 14 rows
// recomputes 4 of its 18 rows instead of 4 of 8.  Measured per step: 1000 x 100 channel 6.6 us
// (strip kernel 18.5 at its best tiling, the one-column kernel before it 23), 600 x 80 5.4 us (17.8;
// 28), with bubbles 5.8, 251 x 190 periodic 5.2 us (19.0; 23), 100 x 50 5.0 us, isothermal 3.8.  What is left on 1000 x 100 (cycles at
// 2.07 GHz, one tile's trace): 1300 until the tiles around are seen done, 2000 to 3000 for 92 KB of
// populations from L2, 1300 for phase A, 1500 for B, 700 for C, 1200 until the stores are counted.
//
// Between steps there is no grid barrier, and nothing that a row does not need is on its path: a
// warp polls the done counts of the tiles around its own (one lane per tile), and each warp adds to
// its tile's count as soon as its own stores are out.  Two more warps per CTA, without a row, serve
// the others.  The first waits for the mass total of the step before (Eq. 14), whose mean density is
// exactly the one that one launch per step uses and is needed only before the force, then adds the
// tile's sums to the instance's fixed-point totals, the mass first, right after phase A, so that the
// total is complete long before the next step's force.  The second writes the record of a step whose
// last tile this was (some microseconds of dependent loads and FP64, which would hold up the next
// step if a warp on that path did it).  Every wait is bounded as in overlapped_steps; all CTAs are
// resident (cooperative launch) and run their tiles in step order, so a wait is always for work
// that some CTA is free to do.
#pragma once

#include "lbm_lane.cuh"

namespace pplbm {

constexpr int FLAT_MAX_ROWS = 14;                  // output rows per tile
constexpr int FLAT_MAX_WARPS = FLAT_MAX_ROWS + 6;  // with the halo rows' warps and the two without a row
constexpr int FLAT_WIDTH = 60;                     // output columns per tile, at most
constexpr int FLAT_MAX_ROUNDS = 8;                  // tiles per CTA, at most
// Registers per thread: 20 warps, one CTA of 14 rows or two of 4, fill the register files of an SM
// (five warps of 96 registers in each quarter's 16384).
constexpr int FLAT_REGS = 96;

// Shared memory per row: psi (the pair, east minus west, east plus west) and u_act,y; density and
// temperature deviations for the totals (of two steps); the pulled g, and for tau_f != 1 the pulled f
// (each lane's own, held there between the phases).
// Then, in launches over several instances, the descriptors of the CTA's tiles.
__host__ __device__ constexpr size_t flat_rows_bytes(bool relax_f, int warps) {
  return sizeof(float2) * 32 * (size_t)(warps - 2) * (8 + 9 + (relax_f ? 9 : 0));
}
inline size_t flat_smem_bytes(int flags, int warps, int insts) {
  return flat_rows_bytes((flags & STEP_RELAX) != 0, warps) + (size_t)insts * sizeof(Inst);
}

// Per row: flux in and out, vapour area, wall, heater and zone vapour.
struct FlatRow {
  float fi, fo, va, wv, hv, zv;
};

struct FlatShared {
  FlatTile tile[FLAT_MAX_ROUNDS];
  long long step0[FLAT_MAX_ROUNDS];
  double rho0[FLAT_MAX_ROUNDS];
  int local0[FLAT_MAX_ROUNDS];
  FlatRow row[2][FLAT_MAX_WARPS];
  double rho[2];
  // a wait of turn t gave up: word t & 1, which nobody writes again before all the turn's warps have read it
  int bad[2];
  // completed steps for the finishing warp, by turns: the instance's position among the CTA's tiles
  // (-1: the launch is over) and the step's number
  int fin_round[2];
  long long fin_step[2];
};
__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
// Sums of two values at once, in the additions of one: a in lanes 0 to 15, b in lanes 16 to 31.
__device__ __forceinline__ double warp_sums(double a, double b) {
  const bool upper = (threadIdx.x & 16) != 0;
  double x = (upper ? b : a) + __shfl_xor_sync(0xffffffffu, upper ? a : b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ long long ld_acquire(const long long* p) {
  long long v;
  asm volatile("ld.acquire.gpu.global.s64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// Polls *p until it reaches need: as flow_wait, each poll an acquire.
__device__ __forceinline__ bool flat_wait(const unsigned* p, unsigned need, const GridBar* bar, unsigned max_polls) {
  const volatile unsigned* const vstatus = &bar->status;
  unsigned polls = 0;
  unsigned long long t0 = 0;
  while (ld_acquire(p) < need) {
    if (polls == 0) t0 = global_ns();
    ++polls;
    __nanosleep(20);  // the line polled is the one being added to
    if ((max_polls != 0 && polls >= max_polls) || ((polls & 15u) == 0 && (*vstatus != 0 || global_ns() - t0 > BARRIER_WAIT_NS)))
      return ld_acquire(p) >= need;
  }
  return true;
}
__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }
// Named barriers: of the rows' warps (1, and 5 once the tiles around are done); of those and the serving warp before the force (2: psi and
// the rows' sums are there, and the mean); after the f collision (3: the rows' warps arrive, the
// serving warp waits for the fluxes); of the serving and the finishing warp (4).
__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// A row's warp: one tile of step k of the launch (step: the instance's step number).  false: a
// wait gave up.
template <bool THERMAL, bool FULL, bool EDGE>
__device__ __forceinline__ bool flat_row(const Inst& I, const StripTile& t, const FlatTile& ft, int self, int k, int turn,
                                         long long step, FlatState* fs, unsigned* done, GridBar* bar,
                                         unsigned max_polls, float2* smem, FlatShared& sh) {
  using Step = LaneStep<THERMAL, FULL, EDGE>;
  const Step L(I, t);
  InstState* const st = I.st;
  const int warp = uni((int)(threadIdx.x >> 5)), nrows = (int)(blockDim.x >> 5) - 2, threads = (int)blockDim.x - 32;
  const int rows = t.y1 - t.y0, r = t.y0 - 2 + warp;
  float2* const sC = smem + L.lane;  // row w at [w * 32]
  float2* const sD = sC + 32 * nrows;
  float2* const sS = sD + 32 * nrows;
  float2* const sU = sS + 32 * nrows;
  float2* const sM = sU + 32 * nrows * (1 + 2 * (turn & 1));
  float2* const sE = sM + 32 * nrows;
  float2* const sG = sU + 32 * nrows * 5 + warp * 9 * 32;
  float2* const sF = sU + 32 * nrows * 14 + warp * 9 * 32;
  FlatRow& row = sh.row[turn & 1][warp];
  const bool in = warp < rows + 4 && L.row_in(r);
  const bool out = warp >= 2 && warp < rows + 2;
  const int rn = L.row_of(r);
  const float2 zero = make_float2(0.0f, 0.0f);

  // the tiles around this one have finished the step before: the first warp (a halo row, idle since
  // phase B) polls their counts, a lane each
  if (k > 0) {
    if (warp == 0) {
      bool got = true;
      if (L.lane < ft.ndeps)
        got = flat_wait(done + (size_t)ft.deps[L.lane] * FLAT_DONE_STRIDE, (unsigned)k * ft.dep_rows[L.lane], bar,
                        max_polls);
      if (!__all_sync(0xffffffffu, got) && L.lane == 0) *reinterpret_cast<volatile int*>(&sh.bad[turn & 1]) = 1;
    }
    bar_sync(5, threads - 32);
  }

  // ===================== phase A: the warp's row =====================
  typename Step::Node n{zero, zero, zero, zero, zero, zero, zero, zero};
  bool ok = true;
  if (in) {
    float2 pf[9], pg[9];
    L.load_row(r, pf, pg);
    L.fill(rn, step, pf, pg);
    L.node(pf, pg, n, ok);
    if (THERMAL) {
#pragma unroll
      for (int i = 0; i < 9; ++i) sG[i * 32] = pg[i];
    }
    if (t.relax_f) {
#pragma unroll
      for (int i = 0; i < 9; ++i) sF[i * 32] = pf[i];
    }
  }
  const PsiRow M = L.psi_row(n.dpsi);
  sC[warp * 32] = M.c;
  sD[warp * 32] = M.d;
  sS[warp * 32] = M.s;
  if (out) {
    sM[warp * 32] = n.drho;
    if (THERMAL) sE[warp * 32] = n.dT;
    if (L.bubbles) {
      const bool lo = !L.pery && rn == 0;
      const int hx = I.heater_x0, hl = I.heater_len;
      const bool va = L.out_a && n.drho.x < L.C.drho_vapor, vb = L.out_b && n.drho.y < L.C.drho_vapor;
      auto count = [&](bool a, bool b) {
        return (float)(__popc(__ballot_sync(0xffffffffu, a)) + __popc(__ballot_sync(0xffffffffu, b)));
      };
      const bool za = L.ca >= hx - hl && L.ca < hx + 2 * hl, zb = L.cb >= hx - hl && L.cb < hx + 2 * hl;
      const bool ha = L.ca >= hx && L.ca < hx + hl, hb = L.cb >= hx && L.cb < hx + hl;
      const float v = count(va, vb), z = count(va && za, vb && zb), h = count(va && ha, vb && hb);
      if (L.lane == 0) {
        row.va = v;
        row.zv = z;
        row.wv = lo ? v : 0.0f;
        row.hv = lo ? h : 0.0f;
      }
    }
    if (L.hazi) L.history(rn, n);
    L.probes(rn, n, [&](int j, float p) { *reinterpret_cast<volatile double*>(&fs->slot[step & 3].probe[j]) = (double)p; });
  }
  if (L.bad(ok)) atomicOr(&st->status, STATUS_UNSTABLE);
  bar_sync(2, threads);
  if (*reinterpret_cast<volatile int*>(&sh.bad[turn & 1])) return false;

  // ===================== phase B: force, u_act, f collision =====================
  typename Step::Flow o;
  float2 dxu = zero;
  if (in && warp >= 1 && warp < rows + 3) {
    PsiRow N{sC[(warp + 1) * 32], sD[(warp + 1) * 32], sS[(warp + 1) * 32]};
    const PsiRow S{sC[(warp - 1) * 32], sD[(warp - 1) * 32], sS[(warp - 1) * 32]};
    if (L.pool && r == L.ny - 1) N = M;  // above the pool's top the ghost row repeats
    o = L.flow(rn, N, M, S, n.drho, n.jx, n.jy, float(I.rho_ref - sh.rho[turn & 1]));
    if (THERMAL) {
      sU[warp * 32] = o.uay;
      float2 E, W;
      L.east_west(o.uax, E, W);
      dxu = v_sub(E, W);
    }
    if (out) {
      if (EDGE && L.channel) {
        float fi = 0.0f, fo = 0.0f;
        if (L.inl_a && L.out_a) fi = __fmaf_rn(0.5f, o.Fx.x, n.jx.x);  // rho u_act = j + F / 2
        if (L.outl_a && L.out_a) fo = __fmaf_rn(0.5f, o.Fx.x, n.jx.x);
        if (L.outl_b && L.out_b) fo = __fmaf_rn(0.5f, o.Fx.y, n.jx.y);
        fi = warp_sum(fi);  // one lane's value: exact
        fo = warp_sum(fo);
        if (L.lane == 0) {
          row.fi = fi;
          row.fo = fo;
        }
      }
      float2 v[9];
      L.collide_f(o, n.drho, n.jx, n.jy, [&](int i) { return sF[i * 32]; }, v);
      L.store_row(t.fout, rn, v);
    }
  }
  bar_arrive(3, threads);
  bar_sync(1, threads - 32);  // u_act is there, and psi may be overwritten

  // ===================== phase C: source and g collision =====================
  if (THERMAL && out) {
    float2 v[9];
    L.collide_g(rn, o.uax, o.uay, sU[(warp + 1) * 32], sU[(warp - 1) * 32], dxu, n.dT, n.coef, n.hm,
                [&](int i) { return sG[i * 32]; }, v);
    L.store_row(t.gout, rn, v);
  }
  if (out) {
    __syncwarp();
    if (L.lane == 0) red_release(done + (size_t)self * FLAT_DONE_STRIDE, 1u);  // the row's populations are written before its count
  }
  return true;
}

// Adds lane j's share x of total j (lanes below NPART; a power of two times FP64: exact) in fixed point.
__device__ __forceinline__ void flat_add(FlatState* fs, int slot, InstState* st, double x) {
  const int lane = threadIdx.x & 31;
  long long q = 0;
  if (fabs(x) < 0x1p62) q = __double2ll_rn(x);
  else atomicOr(&st->status, STATUS_UNSTABLE);
  if (lane < NPART && q != 0) atomicAdd(&fs->slot[slot].sums[lane], (unsigned long long)q);
}

// The serving warp's part of a tile: the mean density of the step before for the rows' warps, then
// the tile's sums.  done: the tile was the step's last.
template <bool THERMAL, bool FULL>
__device__ __forceinline__ bool flat_serve(const Inst& I, const StripTile& t, const FlatTile& ft, int k, int turn,
                                           long long step, double rho_first, FlatState* fs, GridBar* bar,
                                           unsigned max_polls, const float2* smem, FlatShared& sh, bool& done) {
  const int lane = threadIdx.x & 31, nrows = (int)(blockDim.x >> 5) - 2, threads = (int)blockDim.x - 32;
  InstState* const st = I.st;
  const int rows = t.y1 - t.y0;
  const int slot = (int)(step & 3), slot_prev = (int)((step - 1) & 3);
  double rho = rho_first;
  bool got = true;
  if (k > 0) {
    // this step's slot: its totals of four steps back have been taken and cleared (first: the other
    // wait is the longer one)
    const long long cleared = step - 2 < step - k ? step - k : step - 2;
    if (ld_acquire(&st->step) < cleared) {
      unsigned polls = 0;
      got = flow_wait<long long>(&st->step, cleared, bar, max_polls, polls, global_ns());
      fence_gpu();  // the clears are seen before this tile adds
    }
    if (got) got = flat_wait(&fs->slot[slot_prev].count, (unsigned)ft.ntiles, bar, max_polls);
    // as finish_step forms it: the same totals give the same mean
    const double nn = (double)I.nx * (double)I.ny;
    const long long m = *reinterpret_cast<const volatile long long*>(&fs->slot[slot_prev].sums[0]);
    rho = ((double)m * I.fix_unscale[0] + nn * I.rho_ref) / nn;
  }
  if (lane == 0) {
    if (!got) *reinterpret_cast<volatile int*>(&sh.bad[turn & 1]) = 1;
    sh.rho[turn & 1] = rho;
  }
  __syncwarp();
  bar_sync(2, threads);
  if (*reinterpret_cast<volatile int*>(&sh.bad[turn & 1])) return false;

  // the mass, which every tile of the next step waits for
  const bool pery = t.geometry == GEOM_PERIODIC, channel = t.geometry == GEOM_CHANNEL;
  const bool bubbles = FULL && I.bubble_stats != 0;
  const float2* const sM = smem + lane + 32 * nrows * (4 + 2 * (turn & 1));
  const float2* const sE = sM + 32 * nrows;
  const bool out_a = lane >= 1 && lane <= t.wout / 2 && t.xs + 2 * lane < t.nx, out_b = out_a && t.xs + 2 * lane + 1 < t.nx;
  // A lane's two columns over the tile's rows: four rows at a time in FP32 (the lowest bands of the
  // other kernels), those sums with their rounding errors summed beside them (Knuth's two-sum), about
  // 48 bits in all.  An FP64 addition takes the warp 64 cycles, and every instruction here waits among
  // the rows' warps on the way to the mass that every tile waits for: 1000 x 100 6.62 us a step, 1500 x
  // 150 13.0, 600 x 80 with bubbles 5.74; with the errors of every row 6.82, 13.5 and 5.84, and rolled
  // loops of four or seven rows 7.3 to 7.5, 15.2 and 6.7.
  auto pair_sum = [&](float2 s, float2 c) {
    if (!out_a) s.x = c.x = 0.0f;
    if (!out_b) s.y = c.y = 0.0f;
    const float h = __fadd_rn(s.x, s.y), z = __fsub_rn(h, s.x);
    const float e = __fadd_rn(__fsub_rn(s.x, __fsub_rn(h, z)), __fsub_rn(s.y, z));
    return (double)h + (double)__fadd_rn(e, __fadd_rn(c.x, c.y));
  };
  auto column_sum = [&](const float2* v) {
    float2 s = make_float2(0.0f, 0.0f), c = s;
    float2 a = s;
    auto take = [&] {
      const float2 h = v_add(s, a), z = v_sub(h, s);
      c = v_add(c, v_add(v_sub(s, v_sub(h, z)), v_sub(a, z)));
      s = h;
    };
#pragma unroll
    for (int w = 0; w < FLAT_MAX_ROWS; ++w) {
      if (w >= rows) break;
      a = w % 4 == 0 ? v[(w + 2) * 32] : v_add(a, v[(w + 2) * 32]);
      if (w == 3) s = a;
      else if (w % 4 == 3) take();
    }
    if (rows % 4 != 0) take();
    return pair_sum(s, c);
  };
  const double scale = I.fix_scale[lane < NPART ? lane : 0];
  const double mass = warp_sum(column_sum(sM));
  flat_add(fs, slot, st, lane == 0 ? mass * scale : 0.0);
  if (lane == 0) {
    fence_gpu();  // the addition is performed before the count
    atomicAdd(&fs->slot[slot].count, 1u);
  }
  __syncwarp();

  // the other sums, the fluxes through the open ends among them, then the count of complete tiles
  const FlatRow* const all = sh.row[turn & 1];
  const FlatRow& row = all[2 + (lane < rows ? lane : 0)];
  const bool mine = lane < rows;
  double x = 0.0;
  if (THERMAL) {
    const double energy = column_sum(sE);
    if (!pery && t.y0 == 0) {  // with the heater row
      const int ca = t.xs + 2 * lane, hx0 = I.heater_x0, hx1 = hx0 + I.heater_len;
      float2 h = sE[2 * 32];
      if (ca < hx0 || ca >= hx1) h.x = 0.0f;
      if (ca + 1 < hx0 || ca + 1 >= hx1) h.y = 0.0f;
      const double both = warp_sums(energy, pair_sum(h, make_float2(0.0f, 0.0f)));
      const double heat = __shfl_sync(0xffffffffu, both, 16);
      if (lane == 1) x = both;
      if (lane == 2) x = heat;
    } else {
      const double sum = warp_sum(energy);
      if (lane == 1) x = sum;
    }
  }
  if (bubbles) {
    const float va = warp_sum(mine ? row.va : 0.0f), wv = warp_sum(mine ? row.wv : 0.0f);  // counts: exact
    const float hv = warp_sum(mine ? row.hv : 0.0f), zv = warp_sum(mine ? row.zv : 0.0f);
    if (lane == 5) x = (double)va;
    if (lane == 6) x = (double)wv;
    if (lane == 7) x = (double)hv;
    if (lane == 8) x = (double)zv;
  }
  bar_sync(3, threads);
  if (channel && (t.xs < 1 || t.xs + t.wout + 3 > t.nx - 2)) {
    const double both = warp_sums(mine ? (double)row.fi : 0.0, mine ? (double)row.fo : 0.0);
    const double fo = __shfl_sync(0xffffffffu, both, 16);
    if (lane == 3) x = both;
    if (lane == 4) x = fo;
  }
  flat_add(fs, slot, st, x * scale);
  fence_gpu();
  __syncwarp();
  unsigned ticket = 0;
  if (lane == 0) ticket = atomicAdd(&fs->slot[slot].complete, 1u);
  done = __shfl_sync(0xffffffffu, ticket, 0) == (unsigned)(ft.ntiles - 1);
  return true;
}

// The finishing warp: a step whose last tile this CTA had.  Its record, mean density and step count;
// every tile has read the mass total of the step before, whose slot is cleared.
template <bool THERMAL>
__device__ __forceinline__ void flat_finish(const Inst& I, FlatState* fs, long long step, GridBar* bar,
                                            unsigned max_polls) {
  const int lane = threadIdx.x & 31;
  const int slot = (int)(step & 3), slot_prev = (int)((step - 1) & 3);
  InstState* const st = I.st;
  unsigned polls = 0;
  // in step order (another CTA may still be at the step before)
  if (!flow_wait<long long>(&st->step, step, bar, max_polls, polls, global_ns())) {
    if (lane == 0) {
      atomicOr(&bar->status, 1u);
      atomicOr(&st->status, STATUS_TIMEOUT);
    }
    return;
  }
  __threadfence();
  double x = 0.0;
  if (lane < NPART) {
    x = (double)*reinterpret_cast<const volatile long long*>(&fs->slot[slot].sums[lane]) * I.fix_unscale[lane];
    fs->slot[slot_prev].sums[lane] = 0ull;
  }
  double tot[NPART];
#pragma unroll
  for (int j = 0; j < NPART; ++j) tot[j] = __shfl_sync(0xffffffffu, x, j);
  __threadfence();  // every lane's clears are performed before the step count, after which the slot is used again
  __syncwarp();
  if (lane == 0) {
    fs->slot[slot_prev].count = 0u;
    fs->slot[slot_prev].complete = 0u;
    st->p_probe[2 * (step & 1)] = *reinterpret_cast<const volatile double*>(&fs->slot[slot].probe[0]);
    st->p_probe[2 * (step & 1) + 1] = *reinterpret_cast<const volatile double*>(&fs->slot[slot].probe[1]);
    finish_step<THERMAL, MODE_STEP>(I, st, tot, step);  // fences before it publishes the step count
  }
  __syncwarp();
}

template <bool THERMAL, bool FULL, bool PCONST>
__global__ void __maxnreg__(FLAT_REGS)
lbm_flat_kernel(const Inst* __restrict__ insts, const FlatTile* __restrict__ tiles, int ntiles, int nsteps,
                FlatState* fstate, unsigned* done, GridBar* bar, unsigned max_polls, int relax_f,
                const __grid_constant__ Inst kI) {
  extern __shared__ __align__(16) float2 flat_smem[];
  __shared__ FlatShared sh;
  // this CTA's tiles, and what their instances' states are before the launch changes them (no
  // step can complete before this CTA has run its tiles of it)
  const int rounds = (ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
  for (int i = threadIdx.x; i < rounds * (int)(sizeof(FlatTile) / 4); i += blockDim.x) {
    const int rd = i / (int)(sizeof(FlatTile) / 4), w = i - rd * (int)(sizeof(FlatTile) / 4);
    reinterpret_cast<int*>(&sh.tile[rd])[w] =
        reinterpret_cast<const int*>(tiles + blockIdx.x + (size_t)rd * gridDim.x)[w];
  }
  if (threadIdx.x == 0) sh.bad[0] = sh.bad[1] = 0;
  __syncthreads();
  if ((int)threadIdx.x < rounds) {
    const int rd = threadIdx.x;
    const InstState* const st = PCONST ? kI.st : insts[sh.tile[rd].inst].st;
    const long long s0 = *reinterpret_cast<const volatile long long*>(&st->step);
    sh.step0[rd] = s0;
    sh.rho0[rd] = *reinterpret_cast<const volatile double*>(&st->rho_avg[(s0 - 1) & 1]);
    sh.local0[rd] = *reinterpret_cast<const volatile int*>(&st->local_read);
  }
  Inst* const held = reinterpret_cast<Inst*>(reinterpret_cast<char*>(flat_smem) +
                                             flat_rows_bytes(relax_f != 0, (int)(blockDim.x >> 5)));
  if constexpr (!PCONST) {
    for (int rd = 0; rd < rounds; ++rd) {
      const int* src = reinterpret_cast<const int*>(insts + sh.tile[rd].inst);
      int* dst = reinterpret_cast<int*>(held + rd);
      for (int i = threadIdx.x; i < (int)(sizeof(Inst) / 4); i += blockDim.x) dst[i] = src[i];
    }
  }
  __syncthreads();
  const int warp = (int)(threadIdx.x >> 5), nwarps = (int)(blockDim.x >> 5);
  if (warp == nwarps - 1) {
    for (int msg = 0;; msg ^= 1) {
      bar_sync(4, 64);
      const int rd = *reinterpret_cast<volatile int*>(&sh.fin_round[msg]);
      if (rd < 0) return;
      const long long step = *reinterpret_cast<volatile long long*>(&sh.fin_step[msg]);
      const Inst* Ip;
      if constexpr (PCONST) Ip = &kI;
      else Ip = held + rd;
      flat_finish<THERMAL>(*Ip, fstate + sh.tile[rd].inst, step, bar, max_polls);
    }
  }
  const bool serving = warp == nwarps - 2;
  bool go = true;
  int turn = 0, msg = 0;
  for (int k = 0; k < nsteps && go; ++k) {
    for (int rd = 0; rd < rounds && go; ++rd, ++turn) {
      const FlatTile& ft = sh.tile[rd];
      const Inst* Ip;
      if constexpr (PCONST) Ip = &kI;
      else Ip = held + rd;
      const Inst& I = *Ip;
      const long long step = sh.step0[rd] + k;
      const int self = (int)blockIdx.x + rd * (int)gridDim.x;
      StripTile t;
      strip_tile_consts<PCONST>(t, I, uni((int)(step & 1)), k == 0 && sh.local0[rd] != 0, false);
      t.xs = uni(ft.x0) - 2;
      t.wout = uni((int)ft.wout);
      t.y0 = uni(ft.y0);
      t.y1 = t.y0 + uni(ft.rows);
      FlatState* const fs = fstate + ft.inst;
      if (serving) {
        bool last = false;
        go = flat_serve<THERMAL, FULL>(I, t, ft, k, turn, step, sh.rho0[rd], fs, bar, max_polls, flat_smem, sh, last);
        if (last) {
          // waits until the finishing warp is free
          if ((threadIdx.x & 31) == 0) {
            sh.fin_round[msg] = rd;
            sh.fin_step[msg] = step;
          }
          msg ^= 1;
          __syncwarp();
          bar_sync(4, 64);
        }
      } else if (t.xs >= 1 && t.xs + t.wout + 3 <= t.nx - 2) {
        go = flat_row<THERMAL, FULL, false>(I, t, ft, self, k, turn, step, fs, done, bar, max_polls, flat_smem, sh);
      } else {
        go = flat_row<THERMAL, FULL, true>(I, t, ft, self, k, turn, step, fs, done, bar, max_polls, flat_smem, sh);
      }
      if (!go && (threadIdx.x & 31) == 0) {
        atomicOr(&bar->status, 1u);
        atomicOr(&I.st->status, STATUS_TIMEOUT);
      }
    }
  }
  if (serving) {
    if ((threadIdx.x & 31) == 0) sh.fin_round[msg] = -1;
    __syncwarp();
    bar_sync(4, 64);
  }
}

// ---------------------------------------------------------------------------
// Host launchers.
// ---------------------------------------------------------------------------
template <typename Kernel>
cudaError_t flat_set_smem_limit(Kernel fn) {
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)flat_smem_bytes(STEP_RELAX, FLAT_MAX_WARPS, FLAT_MAX_ROUNDS));
}
template <typename Kernel>
int flat_resident(Kernel fn, int flags, int warps, int insts) {
  int n = 0;
  if (flat_set_smem_limit(fn) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, 32 * warps, flat_smem_bytes(flags, warps, insts)) !=
          cudaSuccess)
    return 0;
  return n;
}

template <bool THERMAL, typename Use>
auto flat_kernel_for(int flags, bool single, const Use& use) {
  const bool full = (flags & STEP_FULL) != 0;
  if (full) return single ? use(lbm_flat_kernel<THERMAL, true, true>) : use(lbm_flat_kernel<THERMAL, true, false>);
  return single ? use(lbm_flat_kernel<THERMAL, false, true>) : use(lbm_flat_kernel<THERMAL, false, false>);
}

}  // namespace pplbm
