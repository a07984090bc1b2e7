// FP32 step with one warp per strip of columns and two adjacent columns per lane.
//
// The same time step as lbm_fused_kernel (Sec. 2 of Mukherjee, Basu & Mondal, arXiv 2009.05264,
// with the boundary conditions of Sec. 2.C), organised so that no warp waits for another: a warp
// owns a strip of at most 60 output columns and marches up its band of rows; lane l holds the
// nodes xs + 2 l and xs + 2 l + 1 of a row (xs two columns left of the strip), so every
// arithmetic instruction is a packed FP32 one (FADD2 / FMUL2 / FFMA2) for two nodes, the
// east and west neighbours of psi and u_act come from the adjacent lanes by shuffles, and the rows
// around a node are the warp's own previous iterations.  At iteration k the warp holds the
// pulled populations of row r = y0 - 2 + k (phase A: boundary fill, moments, EOS, psi), does
// force, u_act and the f collision of row r - 1 (phase B) and the g collision of row r - 2
// (phase C).  There is no barrier in the loop.
//
// Why this shape: the one-column kernel's step took 20.9 warp-instructions per node, two
// barriers per row and 18 four-byte asynchronous copies per node, and was bound by their
// latency at four warps per scheduler with neither DRAM nor any pipe busy.  Two nodes per lane
// halve the instructions of everything (13.2 warp-instructions per node in the overlapped loop, its
// waits included), the shuffles replace the
// shared-memory rings of psi and u_act, and without barriers the loads of row r + 1, issued
// between phases A and B into registers, have the rest of the iteration to arrive.  A warp loses
// 4 of its 64 columns to the halo, as much as a 128-column CTA did.  8000 x 800 channel: 172 to
// 176 us a step (36.4 to 37.2 GLUPS; 156 B of DRAM traffic a node, 5.7 TB/s = 0.84 of the copy
// rate) against 196; issue active 28 %, the warps mostly wait for their loads.  Tried and slower: the rows staged in shared
// memory by 16-byte cp.async (204 us), the loop unrolled by 2 or 3 (194, 254: spills),
// 144 registers for 14 warps per SM (283, spills), 184 for 10 (197).
//
// Layout requirement: even row pitch and plane size and 8-byte aligned population buffers (the
// library's own layout).  lbm_step_noalloc's caller layouts use the one-column kernel.
#pragma once

#include "lbm_lane.cuh"

namespace pplbm {

// Warps of a tile of `cols` - 8 output columns and the columns each of them writes (the last one
// what is left): one warp of 56, two of 60, five of 50.
__host__ __device__ constexpr int strip_warps(int cols) { return (cols - 8 + 59) / 60; }
__host__ __device__ constexpr int strip_width(int cols) {
  return ((cols - 8 + strip_warps(cols) - 1) / strip_warps(cols) + 1) / 2 * 2;
}
constexpr int STRIP_MAX_WARPS = 5;

// Shared memory: each lane's own staged populations (never read by another lane): g of three rows
// (between phases A and C) and f of two rows (between A and B; only read for tau_f != 1), per
// warp [slot][population][lane].
constexpr int SF_SLOTS = 2;
constexpr int SG_SLOTS = 3;
__host__ __device__ constexpr int strip_warp_slots(bool thermal, bool relax_f) {
  return (thermal ? SG_SLOTS : 0) + (relax_f ? SF_SLOTS : 0);
}
inline size_t strip_smem_bytes(int thermal, int flags, int warps) {
  return sizeof(float2) * (size_t)(32 * warps) * 9 * strip_warp_slots(thermal != 0, (flags & STEP_RELAX) != 0);
}

// Kernel parameter of a launch over one instance.
struct StripParams {
  Inst I;
};

// Per-lane sums of a tile (output nodes only: the caller drops the other lanes' at the end).
struct StripSums {
  float2 m, e;
  double h, open;
  float fi, fo, va, wv, hv, zv;
  bool bad;
};

// One warp's share of a tile: output columns [xs + 2, xs + 2 + wout), rows [y0, y1).
template <bool THERMAL, bool FULL, bool EDGE>
__device__ __forceinline__ void strip_rows(const Inst& I, const StripTile& t, float rra, long long step, float2* smem,
                                           StripSums& S) {
  using Step = LaneStep<THERMAL, FULL, EDGE>;
  const Step L(I, t);
  float2* const ringG = smem + L.lane;                                       // [(slot * 9 + i) * 32]
  float2* const ringF = smem + (THERMAL ? SG_SLOTS * 9 * 32 : 0) + L.lane;
  const int ny = t.ny, y0 = t.y0, y1 = t.y1;
  const int kend = y1 - y0 + 4;
  const float2 zero = make_float2(0.0f, 0.0f);
  float2 pf[9], pg[9];  // pulled populations of the next row
#pragma unroll
  for (int i = 0; i < 9; ++i) pf[i] = pg[i] = zero;
  // row r: density deviation, momentum, temperature deviation, source factor; _p row r - 1, _q row r - 2
  typename Step::Node n{zero, zero, zero, zero, zero, zero, zero, zero};
  float2 drho_p = zero, jx_p = zero, jy_p = zero, dT_p = zero, coef_p = zero, hm_p = zero;
  float2 dT_q = zero, coef_q = zero, hm_q = zero;
  PsiRow psM = {zero, zero, zero}, psS = {zero, zero, zero};  // psi of rows r - 1 and r - 2
  // u_act of row r - 1, r - 2 (p) and r - 3 (q); dxu: u_x of the east node minus the west one's
  float2 uax = zero, uay = zero, dxu = zero, uax_p = zero, dxu_p = zero, uay_p = zero, uay_q = zero;
  bool ok = true;
  float2 *gA = ringG, *gB = ringG + 9 * 32, *gC = ringG + 18 * 32;  // g of rows r, r - 2, r - 1
  float2 *fA = ringF, *fB = ringF + 9 * 32;                          // f of rows r, r - 1

  L.load_row(y0 - 2, pf, pg);
#pragma unroll 1
  for (int k = 0; k < kend; ++k) {
    const int r = y0 - 2 + k;
    const int rn = L.row_of(r);
    float2 dpsi = zero;

    // ===================== phase A: row r =====================
    if (L.row_in(r)) {
      L.fill(rn, step, pf, pg);
      L.node(pf, pg, n, ok);
      dpsi = n.dpsi;
      if (THERMAL) {
#pragma unroll
        for (int i = 0; i < 9; ++i) gA[i * 32] = pg[i];
      }
      if (t.relax_f) {
#pragma unroll
        for (int i = 0; i < 9; ++i) fA[i * 32] = pf[i];
      }
      if (r >= y0 && r < y1) {
        const bool lo = !L.pery && rn == 0;
        S.m = v_add(S.m, n.drho);
        if (THERMAL) {
          S.e = v_add(S.e, n.dT);
          if (lo) {
            const float2 h = L.heater_dT(n.dT);
            S.h = (double)h.x + (double)h.y;
          }
        }
        if (L.bubbles) {
          const int hx = I.heater_x0, hl = I.heater_len;
          const float va = L.out_a && n.drho.x < L.C.drho_vapor ? 1.0f : 0.0f;
          const float vb = L.out_b && n.drho.y < L.C.drho_vapor ? 1.0f : 0.0f;
          S.va += va + vb;
          if (L.ca >= hx - hl && L.ca < hx + 2 * hl) S.zv += va;
          if (L.cb >= hx - hl && L.cb < hx + 2 * hl) S.zv += vb;
          if (lo) {
            S.wv += va + vb;
            if (L.ca >= hx && L.ca < hx + hl) S.hv += va;
            if (L.cb >= hx && L.cb < hx + hl) S.hv += vb;
          }
        }
        if (L.hazi) L.history(rn, n);
        L.probes(rn, n, [&](int j, float p) { st_probe(I.st, 2 * (int)(step & 1) + j, p); });
        if (EDGE && t.post_open && !L.local && (L.inl_a || L.outl_a || L.outl_b)) S.open += L.open_mass(rn, pf);
      }
    }

    // the next row's loads fly during phases B and C
    if (k + 1 < kend) L.load_row(r + 1, pf, pg);

    // rows outside the lattice are solid (zero); above the pool's top the ghost row repeats
    PsiRow psN = L.psi_row(dpsi);
    if (L.pool && r == ny) psN = psM;

    // ===================== phase B: row q = r - 1 =====================
    const int q = r - 1;
    if (q >= y0 - 1 && L.row_in(q)) {
      const typename Step::Flow o = L.flow(q, psN, psM, psS, drho_p, jx_p, jy_p, rra);
      uax = o.uax;
      uay = o.uay;
      if (THERMAL) {
        float2 E, W;
        L.east_west(uax, E, W);
        dxu = v_sub(E, W);
      }
      if (q >= y0 && q < y1) {
        float2 v[9];
        L.collide_f(o, drho_p, jx_p, jy_p, [&](int i) { return fB[i * 32]; }, v);
        L.store_row(t.fout, q, v);
        if (EDGE && L.channel) {  // flux records, rho u_act = j + F / 2
          if (L.inl_a && L.out_a) S.fi += __fmaf_rn(0.5f, o.Fx.x, jx_p.x);
          if (L.outl_a && L.out_a) S.fo += __fmaf_rn(0.5f, o.Fx.x, jx_p.x);
          if (L.outl_b && L.out_b) S.fo += __fmaf_rn(0.5f, o.Fx.y, jx_p.y);
        }
      }
    }

    // ===================== phase C: row q2 = r - 2 =====================
    if (THERMAL) {
      const int q2 = r - 2;
      if (q2 >= y0) {
        float2 v[9];
        L.collide_g(q2, uax_p, uay_p, uay, uay_q, dxu_p, dT_q, coef_q, hm_q, [&](int i) { return gB[i * 32]; }, v);
        L.store_row(t.gout, q2, v);
      }
      float2* const g = gA;  // the next row takes the slot of row r - 2
      gA = gB;
      gB = gC;
      gC = g;
    }
    float2* const f = fA;
    fA = fB;
    fB = f;

    dT_q = dT_p;
    coef_q = coef_p;
    if (L.hazi) hm_q = hm_p;
    drho_p = n.drho;
    jx_p = n.jx;
    jy_p = n.jy;
    dT_p = n.dT;
    coef_p = n.coef;
    if (L.hazi) hm_p = n.hm;
    uay_q = uay_p;
    uay_p = uay;
    uax_p = uax;
    dxu_p = dxu;
    psS = psM;
    psM = psN;
  }
  S.bad = L.bad(ok);
  // sums of the output nodes only
  if (!L.out_a) S.m.x = S.e.x = 0.0f;
  if (!L.out_b) S.m.y = S.e.y = 0.0f;
}

// Per-CTA shared state: the reduction scratch, and for launches over several instances the
// tile's descriptor.
struct StripSharedCommon {
  double red[STRIP_MAX_WARPS][NPART];
  int last;
};
template <bool PCONST>
struct StripShared : StripSharedCommon {
  Inst I;
};
template <>
struct StripShared<true> : StripSharedCommon {};

// One tile of the step: its warps' strips side by side, then the tile's partial sums.
template <bool THERMAL, bool FULL, bool PCONST>
__device__ __forceinline__ void strip_tile(const Inst* __restrict__ insts, const Tile& tile, int cols,
                                           const StripParams& kp, float2* smem, StripShared<PCONST>& sh,
                                           const TileStep& ts = TileStep{}) {
  if constexpr (!PCONST) {
    __syncthreads();  // the previous tile's readers of the shared constants are done
    const int* src = reinterpret_cast<const int*>(insts + tile.inst);
    int* dst = reinterpret_cast<int*>(&sh.I);
    for (int k = threadIdx.x; k < (int)(sizeof(Inst) / 4); k += blockDim.x) dst[k] = src[k];
    __syncthreads();
  }
  const Inst* Ip;
  if constexpr (PCONST)
    Ip = &kp.I;
  else
    Ip = &sh.I;
  const Inst& I = *Ip;
  InstState* const st = I.st;
  const long long step = ts.step >= 0 ? ts.step : st->step;
  const double rho_avg_prev = ts.step >= 0 ? ts.rho_avg_prev : st->rho_avg[(step - 1) & 1];
  const float rra = float(I.rho_ref - rho_avg_prev);
  const bool post_open = ts.post_open && tile.open_end;
  StripTile t;
  const int par = uni((int)(step & 1)), w = uni((int)(threadIdx.x >> 5));
  strip_tile_consts<PCONST>(t, I, par, ts.step >= 0 ? ts.local : st->local_read != 0, post_open);
  t.y0 = uni(tile.y0);
  t.y1 = uni(tile.y1);
  const int width = strip_width(cols), x0 = uni(tile.x0) + w * width;
  t.wout = strip_columns(min(width, cols - 8 - w * width), t.nx - x0);
  t.xs = x0 - 2;
  float2* const ring = smem + w * 32 * 9 * strip_warp_slots(THERMAL, t.relax_f != 0);
  StripSums S{};
  if (t.xs + 2 < t.nx) {  // the last tile of a row may need fewer warps
    // every pulled column in [1, nx - 2]: no open end, no wrap
    if (t.xs >= 1 && t.xs + t.wout + 3 <= t.nx - 2)
      strip_rows<THERMAL, FULL, false>(I, t, rra, step, ring, S);
    else
      strip_rows<THERMAL, FULL, true>(I, t, rra, step, ring, S);
  }
  if (S.bad) atomicOr(&st->status, STATUS_UNSTABLE);
  const double acc[NPART] = {(double)S.m.x + (double)S.m.y, (double)S.e.x + (double)S.e.y, S.h,
                             (double)S.fi, (double)S.fo, (double)S.va, (double)S.wv, (double)S.hv, (double)S.zv};
  if (!FULL && tile.interior)
    post_partials<STRIP_MAX_WARPS, THERMAL, MODE_STEP, 3>(I, st, tile, acc, sh.red, &sh.last, step);
  else
    post_partials<STRIP_MAX_WARPS, THERMAL, MODE_STEP>(I, st, tile, acc, sh.red, &sh.last, step, post_open, S.open);
}

// Registers per thread: 6 CTAs of 64 threads (12 warps) per SM.
constexpr int STRIP_REGS = 168;

template <bool THERMAL, bool FULL, bool PCONST>
__global__ void __maxnreg__(STRIP_REGS)
lbm_strip_kernel(const Inst* __restrict__ insts, const Tile* __restrict__ tiles, int cols,
                 const __grid_constant__ StripParams kp) {
  extern __shared__ __align__(16) float2 strip_smem[];
  __shared__ StripShared<PCONST> sh;
  strip_tile<THERMAL, FULL, PCONST>(insts, tiles[blockIdx.x], cols, kp, strip_smem, sh);
}

// nsteps steps in one cooperative launch, as lbm_persistent_kernel: overlapped steps, or a CTA
// per tile (or tiles drawn from a counter) with a grid barrier between steps.
template <bool THERMAL, bool FULL, bool PCONST>
__global__ void __maxnreg__(STRIP_REGS)
lbm_strip_persistent_kernel(const Inst* __restrict__ insts, const Tile* __restrict__ tiles, int ntiles, int cols,
                            int nsteps, GridBar* bar, unsigned max_polls, const __grid_constant__ StripParams kp,
                            const __grid_constant__ FlowPlan flow) {
  extern __shared__ __align__(16) float2 strip_smem[];
  __shared__ StripShared<PCONST> sh;
  __shared__ int s_tile, s_ok;
  if (flow.enabled) {
    overlapped_steps(insts, PCONST ? &kp.I : nullptr, tiles, ntiles, nsteps, bar, max_polls, flow,
                     [&](const Tile& tile, const TileStep& ts) {
                       strip_tile<THERMAL, FULL, PCONST>(insts, tile, cols, kp, strip_smem, sh, ts);
                     });
    return;
  }
  const bool one_wave = ntiles <= (int)gridDim.x;
  int first_inst = -1;
  for (int n = 0; n < nsteps; ++n) {
    if (one_wave) {
      const Tile tile = tiles[blockIdx.x];
      first_inst = tile.inst;
      strip_tile<THERMAL, FULL, PCONST>(insts, tile, cols, kp, strip_smem, sh);
    } else {
      if (blockIdx.x == 0 && threadIdx.x == 0) bar->next[(n + 1) & 1] = 0u;  // last drawn from in step n - 1
      for (;;) {
        if (threadIdx.x == 0) s_tile = (int)atomicAdd(&bar->next[n & 1], 1u);
        __syncthreads();
        const int t = s_tile;
        __syncthreads();
        if (t >= ntiles) break;
        const Tile tile = tiles[t];
        if (first_inst < 0) first_inst = tile.inst;
        strip_tile<THERMAL, FULL, PCONST>(insts, tile, cols, kp, strip_smem, sh);
        __syncthreads();
      }
    }
    if (n + 1 < nsteps && !grid_barrier(bar, gridDim.x, max_polls, &s_ok)) {
      if (threadIdx.x == 0 && first_inst >= 0) atomicOr(&insts[first_inst].st->status, STATUS_TIMEOUT);
      if (threadIdx.x == 0 && PCONST) atomicOr(&kp.I.st->status, STATUS_TIMEOUT);
      return;
    }
  }
}

// ---------------------------------------------------------------------------
// Host launchers.
// ---------------------------------------------------------------------------
// CTAs of a strip kernel resident per SM (0 on error), after raising its shared-memory limit.
template <typename Kernel>
int strip_resident(Kernel fn, int thermal, int cols, int flags) {
  const int warps = strip_warps(cols);
  const size_t smem = strip_smem_bytes(thermal, flags, warps);
  int n = 0;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)strip_smem_bytes(1, STEP_RELAX, STRIP_MAX_WARPS)) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, 32 * warps, smem) != cudaSuccess)
    return 0;
  return n;
}

template <bool THERMAL>
cudaError_t launch_strip_t(int cols, int flags, const Inst* d_inst, const Tile* d_tiles, int ntiles, cudaStream_t s,
                           const Inst* h_inst) {
  auto go = [&](auto fn, const StripParams& kp) -> cudaError_t {
    const size_t smem = strip_smem_bytes(THERMAL, flags, strip_warps(cols));
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)strip_smem_bytes(1, STEP_RELAX, STRIP_MAX_WARPS));
    if (e != cudaSuccess) return e;
    fn<<<ntiles, 32 * strip_warps(cols), smem, s>>>(d_inst, d_tiles, cols, kp);
    return cudaGetLastError();
  };
  const bool full = (flags & STEP_FULL) != 0;
  StripParams kp{};
  if (!h_inst) return full ? go(lbm_strip_kernel<THERMAL, true, false>, kp) : go(lbm_strip_kernel<THERMAL, false, false>, kp);
  kp.I = *h_inst;
  return full ? go(lbm_strip_kernel<THERMAL, true, true>, kp) : go(lbm_strip_kernel<THERMAL, false, true>, kp);
}

template <bool THERMAL>
cudaError_t launch_strip_persistent_t(int cols, int flags, const Inst* d_inst, const Tile* d_tiles, int ntiles,
                                      int nsteps, GridBar* bar, unsigned max_polls, cudaStream_t s, const Inst* h_inst,
                                      const FlowPlan& flow) {
  auto go = [&](auto fn, const StripParams& kp) -> cudaError_t {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int per_sm = strip_resident(fn, THERMAL, cols, flags);
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ntiles < sms * per_sm ? ntiles : sms * per_sm);
    cfg.blockDim = dim3(32 * strip_warps(cols));
    cfg.dynamicSmemBytes = strip_smem_bytes(THERMAL, flags, strip_warps(cols));
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, d_inst, d_tiles, ntiles, cols, nsteps, bar, max_polls, kp, flow);
  };
  const bool full = (flags & STEP_FULL) != 0;
  StripParams kp{};
  if (!h_inst)
    return full ? go(lbm_strip_persistent_kernel<THERMAL, true, false>, kp)
                : go(lbm_strip_persistent_kernel<THERMAL, false, false>, kp);
  kp.I = *h_inst;
  return full ? go(lbm_strip_persistent_kernel<THERMAL, true, true>, kp)
              : go(lbm_strip_persistent_kernel<THERMAL, false, true>, kp);
}

template <bool THERMAL>
int strip_resident_t(int cols, int flags, bool single, bool persistent) {
  const bool full = (flags & STEP_FULL) != 0;
  if (persistent) {
    if (full) return single ? strip_resident(lbm_strip_persistent_kernel<THERMAL, true, true>, THERMAL, cols, flags)
                            : strip_resident(lbm_strip_persistent_kernel<THERMAL, true, false>, THERMAL, cols, flags);
    return single ? strip_resident(lbm_strip_persistent_kernel<THERMAL, false, true>, THERMAL, cols, flags)
                  : strip_resident(lbm_strip_persistent_kernel<THERMAL, false, false>, THERMAL, cols, flags);
  }
  if (full) return single ? strip_resident(lbm_strip_kernel<THERMAL, true, true>, THERMAL, cols, flags)
                          : strip_resident(lbm_strip_kernel<THERMAL, true, false>, THERMAL, cols, flags);
  return single ? strip_resident(lbm_strip_kernel<THERMAL, false, true>, THERMAL, cols, flags)
                : strip_resident(lbm_strip_kernel<THERMAL, false, false>, THERMAL, cols, flags);
}

}  // namespace pplbm
