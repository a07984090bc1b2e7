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
// halve the instructions of everything (12.1 warp-instructions per node), the shuffles replace the
// shared-memory rings of psi and u_act, and without barriers the loads of row r + 1, issued
// between phases A and B into registers, have the rest of the iteration to arrive.  A warp loses
// 4 of its 64 columns to the halo, as much as a 128-column CTA did.  8000 x 800 channel: 175 us a
// step (36.5 GLUPS, 152 B of DRAM traffic a node = 0.82 of the copy rate) against 196; issue
// active 37 %, the warps mostly wait for their loads.  Tried and slower: the rows staged in shared
// memory by 16-byte cp.async (204 us), the loop unrolled by 2 or 3 (194, 254: spills),
// 144 registers for 14 warps per SM (283, spills), 184 for 10 (197).
//
// Accuracy: the odd part of the f collision takes the momentum and the force themselves, not
// rho u with an approximate 1 / rho, and the rest population closes the node's mass, so the
// velocity error against FP64 is about half the one-column kernel's (3.4e-7 against 1.5e-6 in
// the L2 norm on 1000 x 100 after 500 steps).
//
// All arithmetic of the interior path is written with explicitly rounded operations, so the
// results do not depend on which kernel (one launch per step, persistent, batch) ran it.
//
// Layout requirement: even row pitch and plane size and 8-byte aligned population buffers (the
// library's own layout).  lbm_step_noalloc's caller layouts use the one-column kernel.
#pragma once

#include "lbm_kernels.cuh"

namespace pplbm {

// Warps of a tile of `cols` - 8 output columns and the columns each of them writes (the last one
// what is left): one warp of 56, two of 60, five of 50.
__host__ __device__ constexpr int strip_warps(int cols) { return (cols - 8 + 59) / 60; }
__host__ __device__ constexpr int strip_width(int cols) {
  return ((cols - 8 + strip_warps(cols) - 1) / strip_warps(cols) + 1) / 2 * 2;
}
constexpr int STRIP_MAX_WARPS = 5;
// 3 w of the axis and diagonal links in FP32 (1/3 and 1/12), with 2 B1 + 4 B5 = 1 exactly
constexpr float STRIP_B1 = 0x1.555556p-2f, STRIP_B5 = 0x1.555554p-4f;

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

// ---------------------------------------------------------------------------
// Packed FP32 helpers (x: the lane's first node, y: its second).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 v_bc(float c) { return make_float2(c, c); }
__device__ __forceinline__ float2 v_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 v_sub(float2 a, float2 b) { return __ffma2_rn(b, v_bc(-1.0f), a); }
__device__ __forceinline__ float2 v_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 v_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// MUFU approximations without the denormal scaling around them (at most about 1 ulp; the
// arguments are densities, temperatures and sums of square roots, far from denormal).
__device__ __forceinline__ float s_rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float s_rsqrt(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float s_sqrt(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float2 v_rcp(float2 a) { return make_float2(s_rcp(a.x), s_rcp(a.y)); }
__device__ __forceinline__ float2 v_rsqrt(float2 a) { return make_float2(s_rsqrt(a.x), s_rsqrt(a.y)); }

// Kernel parameter of a launch over one instance.
struct StripParams {
  Inst I;
};

// psi - psi_ref of one row of the warp: the pair itself, east minus west and east plus west.
struct PsiRow {
  float2 c, d, s;
};

// Per-lane sums of a tile (output nodes only: the caller drops the other lanes' at the end).
struct StripSums {
  float2 m, e;
  float h, fi, fo, va, wv, hv, zv;
  double open;
  bool bad;
};

// A value that is the same in every lane, in a form the compiler knows to be so (uniform registers,
// branches and address arithmetic): the descriptor of a single-instance launch is a kernel
// parameter and needs nothing; what comes from memory passes a warp reduction once per tile.
__device__ __forceinline__ int uni(int v) { return (int)__reduce_or_sync(0xffffffffu, (unsigned)v); }
__device__ __forceinline__ char* uni(const void* p) {
  const unsigned long long v = reinterpret_cast<unsigned long long>(p);
  const unsigned lo = __reduce_or_sync(0xffffffffu, (unsigned)v), hi = __reduce_or_sync(0xffffffffu, (unsigned)(v >> 32));
  return reinterpret_cast<char*>((unsigned long long)hi << 32 | lo);
}
// base + i * stride bytes in one wide multiply-add.
__device__ __forceinline__ char* at_plane(char* base, unsigned stride, int i) {
  unsigned long long a;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(a) : "r"(stride), "r"(i), "l"(reinterpret_cast<unsigned long long>(base)));
  return reinterpret_cast<char*>(a);
}

// What strip_rows needs of the tile and of the lattice besides the constants, all uniform.
struct StripTile {
  int nx, ny, pitch, plane, geometry, multiphase;
  const char *fin, *gin;  // populations read
  char *fout, *gout;      // and written
  int xs, wout, y0, y1;   // columns [xs + 2, xs + 2 + wout), rows [y0, y1)
  int local, post_open, relax_f;
};

// One warp's share of a tile: output columns [xs + 2, xs + 2 + wout), rows [y0, y1).
// EDGE: some pulled column lies outside [1, nx - 2] (an open end, a wrap, or beyond the lattice):
// the links then come from per-lane wrapped columns and the nodes at an open end take the
// boundary fill; otherwise only the wall rows (and a pool's top row) differ from the interior.
// FULL: the pool geometry, the Hazi-Markus source and the bubble statistics.
template <bool THERMAL, bool FULL, bool EDGE>
__device__ __forceinline__ void strip_rows(const Inst& I, const StripTile& t, float rra, long long step, float2* smem,
                                           StripSums& S) {
  const KConst<float>& C = I.strip.C;
  const KPair& P = I.strip.P;
  const int lane = threadIdx.x & 31;
  float2* const ringG = smem + lane;                                       // [(slot * 9 + i) * 32]
  float2* const ringF = smem + (THERMAL ? SG_SLOTS * 9 * 32 : 0) + lane;
  const int nx = t.nx, ny = t.ny, xs = t.xs;
  const unsigned plane4 = (unsigned)t.plane * 4u, pitch4 = (unsigned)t.pitch * 4u;
  const bool perx = t.geometry != GEOM_CHANNEL, pery = t.geometry == GEOM_PERIODIC;
  const bool channel = t.geometry == GEOM_CHANNEL;
  const bool pool = FULL && t.geometry == GEOM_POOL;
  const bool multiphase = t.multiphase != 0;
  const bool hazi = FULL && THERMAL && I.source_model == 1;
  const bool bubbles = FULL && I.bubble_stats != 0;
  const bool local = t.local != 0;
  float* const rho_prev = static_cast<float*>(I.rho_prev);
  const int y0 = t.y0, y1 = t.y1;
  const int kend = y1 - y0 + 4;

  // this lane's columns; the strip's halo is two columns a side, lanes beyond it repeat the
  // lane before (their results are not used)
  const int xl = xs + 2 * min(lane, t.wout / 2 + 1);
  int ca = xl, cb = xl + 1, cm = xl - 1, cp = xl + 2;  // columns of the two nodes and beside them
  bool in_a = true, in_b = true;
  if (EDGE) {
    if (perx) {
      ca = wrap_index(xl, nx);
      cb = wrap_index(xl + 1, nx);
      cm = wrap_index(xl - 1, nx);
      cp = wrap_index(xl + 2, nx);
    } else {
      // columns outside the lattice read the end column: a valid state, never used
      in_a = xl >= 0 && xl < nx;
      in_b = xl + 1 >= 0 && xl + 1 < nx;
      ca = min(max(xl, 0), nx - 1);
      cb = min(max(xl + 1, 0), nx - 1);
      cm = min(max(xl - 1, 0), nx - 1);
      cp = min(max(xl + 2, 0), nx - 1);
    }
  }
  const unsigned oa = 4u * ca, ob = 4u * cb, om1 = 4u * cm, op1 = 4u * cp;  // byte offsets in a row
  const bool inl_a = EDGE && channel && xl == 0;  // xs is even: the inlet column is a lane's first node
  const bool outl_a = EDGE && channel && xl == nx - 1, outl_b = EDGE && channel && xl + 1 == nx - 1;
  const bool out_a = lane >= 1 && lane <= t.wout / 2 && xl < nx, out_b = out_a && xl + 1 < nx;

  float2 pf[9], pg[9];  // pulled populations of the next row
#pragma unroll
  for (int i = 0; i < 9; ++i) pf[i] = pg[i] = make_float2(0.0f, 0.0f);

  // bounds-checked builds: byte offset o of plane i against the buffer
  auto fits = [&](const char* buf, const char* p, int bytes) {
    return idx_ok(I.st, p - buf, 9LL * t.plane * 4) && idx_ok(I.st, p - buf + bytes - 1, 9LL * t.plane * 4);
  };
  auto one_at = [&](const char* buf, const char* p) -> float {
    return fits(buf, p, 4) ? *reinterpret_cast<const float*>(p) : 0.0f;
  };
  // populations (row, this lane's nodes shifted by dx columns) of the plane row that starts at p
  auto pair_at = [&](const char* buf, const char* p, int dx) -> float2 {
    if (!EDGE) {
      if (dx == 0) return fits(buf, p + oa, 8) ? *reinterpret_cast<const float2*>(p + oa) : make_float2(0.0f, 0.0f);
      return make_float2(one_at(buf, p + oa + 4 * dx), one_at(buf, p + oa + 4 * dx + 4));
    }
    return make_float2(one_at(buf, p + (dx == 0 ? oa : dx < 0 ? om1 : ob)),
                       one_at(buf, p + (dx == 0 ? ob : dx < 0 ? oa : op1)));
  };
  // loads of row r (nothing for rows outside the lattice)
  auto load_row = [&](int r) {
    if (!pery && (r < 0 || r >= ny)) return;
    const int rn = pery ? wrap_index(r, ny) : r;
    const int rm = rn > 0 ? rn - 1 : ny - 1, rp = rn < ny - 1 ? rn + 1 : 0;  // used unless a wall is there
    const size_t n0 = (size_t)(unsigned)rn * pitch4, nm = (size_t)(unsigned)rm * pitch4, np = (size_t)(unsigned)rp * pitch4;
    const bool lo = !pery && rn == 0, hi = !pery && rn == ny - 1;  // hi: a wall, or the pool's top
    if (!local && !lo && !hi) {
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const size_t o = (size_t)plane4 * i + (lat_cy(i) == 1 ? nm : (lat_cy(i) == -1 ? np : n0));
        pf[i] = pair_at(t.fin, t.fin + o, -lat_cx(i));
        if (THERMAL) pg[i] = pair_at(t.gin, t.gin + o, -lat_cx(i));
      }
    } else {
      // the node's own populations: all of them right after an initialisation, the opposite one
      // for a link from a wall (halfway bounce-back; a pool's top links are set by its fill)
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const bool wall = (lat_cy(i) == 1 && lo) || (lat_cy(i) == -1 && hi);
        if (local || wall) {
          const size_t o = (size_t)plane4 * (local ? i : lat_opp(i)) + n0;
          pf[i] = pair_at(t.fin, t.fin + o, 0);
          if (THERMAL) pg[i] = pair_at(t.gin, t.gin + o, 0);
        } else {
          const size_t o = (size_t)plane4 * i + (lat_cy(i) == 1 ? nm : (lat_cy(i) == -1 ? np : n0));
          pf[i] = pair_at(t.fin, t.fin + o, -lat_cx(i));
          if (THERMAL) pg[i] = pair_at(t.gin, t.gin + o, -lat_cx(i));
        }
      }
    }
  };
  // stores of the nine populations of row y
  auto store_row = [&](char* buf, int y, const float2 (&v)[9]) {
    char* const p = buf + (size_t)(unsigned)y * pitch4 + oa;
    if (!EDGE || out_b) {
      if (out_a) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
          char* const o = at_plane(p, plane4, i);
          if (fits(buf, o, 8)) *reinterpret_cast<float2*>(o) = v[i];
        }
      }
    } else if (out_a) {  // the last column of an odd width
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        char* const o = at_plane(p, plane4, i);
        if (fits(buf, o, 4)) *reinterpret_cast<float*>(o) = v[i].x;
      }
    }
  };

  const float2 zero = make_float2(0.0f, 0.0f);
  // row r: density deviation, momentum, temperature deviation, source factor; _p row r - 1, _q row r - 2
  float2 drho = zero, jx = zero, jy = zero, dT = zero, coef = zero, hm = zero;
  float2 drho_p = zero, jx_p = zero, jy_p = zero, dT_p = zero, coef_p = zero, hm_p = zero;
  float2 dT_q = zero, coef_q = zero, hm_q = zero;
  PsiRow psM = {zero, zero, zero}, psS = {zero, zero, zero};  // psi of rows r - 1 and r - 2
  // u_act of row r - 1, r - 2 (p) and r - 3 (q); dxu: u_x of the east node minus the west one's
  float2 uax = zero, uay = zero, dxu = zero, uax_p = zero, dxu_p = zero, uay_p = zero, uay_q = zero;
  bool ok = true;
  float2 *gA = ringG, *gB = ringG + 9 * 32, *gC = ringG + 18 * 32;  // g of rows r, r - 2, r - 1
  float2 *fA = ringF, *fB = ringF + 9 * 32;                          // f of rows r, r - 1

  load_row(y0 - 2);
#pragma unroll 1
  for (int k = 0; k < kend; ++k) {
    const int r = y0 - 2 + k;
    const bool row_ok = pery || (r >= 0 && r < ny);
    const int rn = pery ? wrap_index(r, ny) : r;
    float2 dpsi = zero;

    // ===================== phase A: row r =====================
    if (row_ok) {
      const bool lo = !pery && rn == 0, hi = !pery && !pool && rn == ny - 1, top = pool && rn == ny - 1;
      if (!local && (lo || hi || top || EDGE)) {
        // boundary nodes, one at a time (wall rows, the pool's top row, open ends)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int xn = h ? cb : ca;
          const NodeBC nb{lo, hi, h == 0 && inl_a, h ? outl_b : outl_a, top};
          if ((h ? in_b : in_a) && (nb.wlo || nb.whi || nb.inl || nb.outl || nb.top)) {
            float f1[9], g1[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) {
              f1[i] = h ? pf[i].y : pf[i].x;
              g1[i] = h ? pg[i].y : pg[i].x;
            }
            if (EDGE || FULL)
              boundary_fill<float, THERMAL>(f1, g1, nb, I, C, reinterpret_cast<const float*>(t.gin), t.plane, t.pitch,
                                            rn * t.pitch + xn, xn, perx, step);
            else if (THERMAL)
              wall_temperature<float>(g1, lo, hi, xn, I, C, step);
#pragma unroll
            for (int i = 0; i < 9; ++i) {
              if (h) {
                pf[i].y = f1[i];
                pg[i].y = g1[i];
              } else {
                pf[i].x = f1[i];
                pg[i].x = g1[i];
              }
            }
          }
        }
      }
      // moments (Eqs. 4, 6, 17)
      const float2 p56 = v_add(pf[5], pf[6]), p78 = v_add(pf[7], pf[8]);
      drho = v_add(v_add(v_add(pf[0], v_add(pf[1], pf[3])), v_add(pf[2], pf[4])), v_add(p56, p78));
      jx = v_add(v_sub(pf[1], pf[3]), v_add(v_sub(pf[5], pf[6]), v_sub(pf[8], pf[7])));
      jy = v_add(v_sub(pf[2], pf[4]), v_sub(p56, p78));
      const float2 rho = v_add(P.rho_ref, drho);
      float2 T = P.T0;
      if (THERMAL) {
        dT = v_add(v_add(v_add(v_add(pg[0], pg[1]), v_add(pg[2], pg[3])),
                         v_add(v_add(pg[4], pg[5]), v_add(pg[6], pg[7]))), pg[8]);
        T = v_add(P.T_ref, dT);
#pragma unroll
        for (int i = 0; i < 9; ++i) gA[i * 32] = pg[i];
      }
      if (t.relax_f) {
#pragma unroll
        for (int i = 0; i < 9; ++i) fA[i * 32] = pf[i];
      }
      ok = ok && rho.x > 0.0f && rho.y > 0.0f;
      float2 drad = zero;
      if (multiphase) {
        // Peng-Robinson (Eq. 12) and psi (Eq. 11) as exact differences from the reference state;
        // with om = 1 - b rho, D = 1 + 2 b rho - (b rho)^2 = 2 - om^2
        const float2 nv = v_fma(P.b, rho, v_bc(-1.0f));
        const float2 om = v_mul(nv, v_bc(-1.0f));
        const float2 invD = v_rcp(v_fma(nv, om, v_bc(2.0f)));
        const float2 inv1 = v_rcp(om);
        float2 z = v_mul(drho, v_mul(v_fma(P.s3, rho, P.rho_ref), invD));
        float2 sa = zero, isT = zero;
        drad = v_mul(v_mul(drho, T), inv1);
        if (THERMAL) {
          // sqrt(alpha) relative to its reference value: 1 + m1 (sqrt T - sqrt T_ref), the
          // difference of the roots as dT / (sqrt T + sqrt T_ref)
          isT = v_rsqrt(T);
          const float2 w = v_mul(dT, v_rcp(v_fma(T, isT, P.sqrtT_r)));
          sa = v_fma(P.m1, w, v_bc(1.0f));
          z = v_mul(v_mul(sa, sa), z);
          drad = v_mul(P.cA, v_fma(P.rho_ref, dT, drad));
          drad = v_fma(P.cB, z, drad);
          drad = v_fma(P.cK, v_mul(w, v_add(sa, v_bc(1.0f))), drad);
        } else {
          drad = v_fma(P.cB, z, v_mul(P.cA, drad));
        }
        drad = v_fma(P.c3, drho, drad);
        const float2 rad = v_add(P.rad_ref, drad);
        const float2 psi = make_float2(s_sqrt(fmaxf(rad.x, 0.0f)), s_sqrt(fmaxf(rad.y, 0.0f)));
        const float2 den = v_add(psi, P.psi_ref);  // zero only where drad is
        dpsi = v_mul(drad, v_rcp(make_float2(fmaxf(den.x, 1e-30f), fmaxf(den.y, 1e-30f))));
        ok = ok && om.x > 0.0f && om.y > 0.0f && rad.x >= 0.0f && rad.y >= 0.0f;
        if (THERMAL) {  // T (1 - (dp/dT)_rho / (rho c_v)) of the second Eq. 19
          const float2 q = v_mul(v_mul(sa, isT), v_mul(rho, invD));
          const float2 Te = v_mul(T, v_fma(P.cR, inv1, v_mul(P.cS, q)));
          coef = v_sub(T, Te);
          if (hazi) {  // first Eq. 19
            coef = T;
            hm = v_mul(Te, v_rcp(rho));
          }
        }
      } else if (THERMAL) {
        coef = T;
        ok = ok && fabsf(T.x) < INFINITY && fabsf(T.y) < INFINITY;
      }
      if (r >= y0 && r < y1) {
        S.m = v_add(S.m, drho);
        if (THERMAL) {
          S.e = v_add(S.e, dT);
          if (lo) {
            if (out_a && ca >= I.heater_x0 && ca < I.heater_x0 + I.heater_len) S.h += dT.x;
            if (out_b && cb >= I.heater_x0 && cb < I.heater_x0 + I.heater_len) S.h += dT.y;
          }
        }
        if (bubbles) {
          const int hx = I.heater_x0, hl = I.heater_len;
          const float va = out_a && drho.x < C.drho_vapor ? 1.0f : 0.0f;
          const float vb = out_b && drho.y < C.drho_vapor ? 1.0f : 0.0f;
          S.va += va + vb;
          if (ca >= hx - hl && ca < hx + 2 * hl) S.zv += va;
          if (cb >= hx - hl && cb < hx + 2 * hl) S.zv += vb;
          if (lo) {
            S.wv += va + vb;
            if (ca >= hx && ca < hx + hl) S.hv += va;
            if (cb >= hx && cb < hx + hl) S.hv += vb;
          }
        }
        if (hazi) {
          // temporal density gradient rho^n - rho^(n-1), both as deviations from rho_ref; this
          // lane owns the nodes' history (read, then overwritten with rho^n)
          const int kp = rn * t.pitch + ca;
          if (out_a && idx_ok(I.st, kp, t.plane)) {
            hm.x = hm.x * (drho.x - rho_prev[kp]);
            rho_prev[kp] = drho.x;
          }
          if (out_b && idx_ok(I.st, kp + 1, t.plane)) {
            hm.y = hm.y * (drho.y - rho_prev[kp + 1]);
            rho_prev[kp + 1] = drho.y;
          }
        }
        if (EDGE && channel && rn == ny / 2) {  // pressure probes
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int xn = h ? cb : ca;
            if ((h ? out_b : out_a) && (xn == 1 || xn == nx - 2)) {
              const float dr = h ? drho.y : drho.x;
              const float p = multiphase ? P.p_ref + ((h ? drad.y : drad.x) * P.inv_ps + dr * (1.0f / 3.0f))
                                         : (h ? rho.y : rho.x) * (1.0f / 3.0f);
              if (xn == 1) st_probe(I.st, 2 * (int)(step & 1), p);
              if (xn == nx - 2) st_probe(I.st, 2 * (int)(step & 1) + 1, p);
            }
          }
        }
        if (EDGE && t.post_open && !local && (inl_a || outl_a || outl_b)) {
          // mass this node's pull took in minus the mass the pull let out of the lattice: in, the
          // open-end links that boundary_fill set; out, this node's post-collision populations
          // that point out of the open end (no node pulls them; at a wall row the diagonal one is
          // bounced back instead)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const bool inl = h == 0 && inl_a, outl = h ? outl_b : outl_a;
            if (!(h ? out_b : out_a)) continue;
            const char* const pn = t.fin + (size_t)rn * pitch4 + (h ? ob : oa);
            auto fl = [&](int i) { return (double)one_at(t.fin, pn + (size_t)plane4 * i); };
            auto fc = [&](int i) { return (double)(h ? pf[i].y : pf[i].x); };
            if (inl)
              S.open += fc(1) + (lo ? 0.0 : fc(5)) + (hi ? 0.0 : fc(8)) - (fl(3) + (hi ? 0.0 : fl(6)) + (lo ? 0.0 : fl(7)));
            else if (outl)
              S.open += fc(3) + (lo ? 0.0 : fc(6)) + (hi ? 0.0 : fc(7)) - (fl(1) + (hi ? 0.0 : fl(5)) + (lo ? 0.0 : fl(8)));
          }
        }
      }
    }

    // the next row's loads fly during phases B and C
    if (k + 1 < kend) load_row(r + 1);

    // psi of row r with its east and west neighbours; rows outside the lattice are solid (zero),
    // above the pool's top the ghost row repeats the row below
    PsiRow psN;
    {
      float w = __shfl_up_sync(0xffffffffu, dpsi.y, 1), e = __shfl_down_sync(0xffffffffu, dpsi.x, 1);
      float ea = dpsi.y;
      if (EDGE) {  // at the open ends the ghost column repeats the end column
        if (inl_a) w = dpsi.x;
        if (outl_a) ea = dpsi.x;
        if (outl_b) e = dpsi.y;
      }
      const float2 E = make_float2(ea, e), W = make_float2(w, dpsi.x);
      psN.c = dpsi;
      psN.d = v_sub(E, W);
      psN.s = v_add(E, W);
      if (pool && r == ny) psN = psM;
    }

    // ===================== phase B: row q = r - 1 =====================
    const int q = r - 1;
    if (q >= y0 - 1 && (pery || (q >= 0 && q < ny))) {
      float2 Fx = zero, Fy = zero;
      if (multiphase) {
        // Eqs. 9, 10, 15: t1 = sum G_i d_i c_i, t2 = sum G_i d_i^2 c_i of d = psi - psi_ref, the
        // squares as products of sums and differences; the diagonal part of t2y is
        // Gh (E_N^2 + W_N^2 - E_S^2 - W_S^2) = Gh / 2 [(s_N - s_S)(s_N + s_S) + (d_N - d_S)(d_N + d_S)]
        const float2 dsum = v_add(psN.d, psS.d);
        const float2 gd = v_mul(P.G2, psM.d);
        const float2 t1x = v_fma(P.Gh, dsum, gd);
        const float2 cdif = v_sub(psN.c, psS.c), sdif = v_sub(psN.s, psS.s);
        const float2 gc = v_mul(P.G2, cdif);
        const float2 t1y = v_fma(P.Gh, sdif, gc);
        const float2 t2x = v_fma(gd, psM.s, v_mul(P.Gh, v_fma(psN.d, psN.s, v_mul(psS.d, psS.s))));
        const float2 m = v_fma(sdif, v_add(psN.s, psS.s), v_mul(v_sub(psN.d, psS.d), dsum));
        const float2 t2y = v_fma(gc, v_add(psN.c, psS.c), v_mul(P.Ghh, m));
        const float2 nlead = v_fma(P.nbeta, psM.c, P.npsi_ref);
        Fx = v_fma(nlead, t1x, v_mul(P.nmix, t2x));
        Fy = v_fma(nlead, t1y, v_mul(P.nmix, t2y));
        if (!pery && q == 0) Fy = v_add(Fy, v_fma(psM.c, P.wall1, P.wall0));
        if (!pery && !pool && q == ny - 1) Fy = v_sub(Fy, v_fma(psM.c, P.wall1, P.wall0));
      }
      Fy = v_fma(v_add(drho_p, v_bc(rra)), P.ng_a, Fy);  // Eq. 14, gravity along -y
      const float2 rho = v_add(P.rho_ref, drho_p);
      const float2 irho = v_rcp(rho);
      const float2 ux = v_mul(jx_p, irho), uy = v_mul(jy_p, irho);
      const float2 dux = v_mul(Fx, irho), duy = v_mul(Fy, irho);
      uax = v_fma(v_bc(0.5f), dux, ux);  // Eq. 7
      uay = v_fma(v_bc(0.5f), duy, uy);
      if (THERMAL) {
        float w = __shfl_up_sync(0xffffffffu, uax.y, 1), e = __shfl_down_sync(0xffffffffu, uax.x, 1);
        float ea = uax.y;
        if (EDGE) {
          if (inl_a) w = uax.x;
          if (outl_a) ea = uax.x;
          if (outl_b) e = uax.y;
        }
        dxu = v_sub(make_float2(ea, e), make_float2(w, uax.x));
      }
      if (q >= y0 && q < y1) {
        // f collision (Eqs. 2, 3, 5), pairwise over opposite directions as in collide_f.  The odd
        // part, 3 w c.(omega rho u + rho du), takes the momentum and the force themselves: the
        // error of the approximate 1 / rho in u would act on the momentum every step.  B1 and B5
        // keep 2 B1 + 4 B5 = 1, and 4.5 w of the axis and diagonal links are exact.
        constexpr float w1 = LatWeights<float>::w1(), w5 = LatWeights<float>::w5();
        const float2 sx = v_fma(v_bc(2.0f), ux, dux), sy = v_fma(v_bc(2.0f), uy, duy);
        const float2 dsx = v_mul(dux, sx), dsy = v_mul(duy, sy);
        const float2 usq = v_fma(ux, ux, v_mul(uy, uy));
        const float2 nr15 = v_mul(v_bc(-1.5f), rho);
        const float2 K = v_fma(nr15, v_add(dsx, dsy), v_mul(P.omega_f, v_fma(nr15, usq, drho_p)));
        const float2 K1 = v_mul(v_bc(w1), K), K5 = v_mul(v_bc(w5), K);
        const float2 a1 = v_mul(v_bc(0.5f), rho), a5 = v_mul(v_bc(0.125f), rho);
        const float2 mx = v_fma(P.omega_f, jx_p, Fx), my = v_fma(P.omega_f, jy_p, Fy);
        float2 v[9];
        auto both = [&](int i, int j, float2 cu, float2 cds, float2 m, float2 a, float b, float2 Kw) {
          const float2 sym = v_fma(a, v_fma(v_mul(P.omega_f, cu), cu, cds), Kw), anti = v_mul(v_bc(b), m);
          v[i] = v_add(sym, anti);
          v[j] = v_sub(sym, anti);
        };
        both(1, 3, ux, dsx, mx, a1, STRIP_B1, K1);
        both(2, 4, uy, dsy, my, a1, STRIP_B1, K1);
        both(5, 7, v_add(ux, uy), v_mul(v_add(dux, duy), v_add(sx, sy)), v_add(mx, my), a5, STRIP_B5, K5);
        both(6, 8, v_sub(uy, ux), v_mul(v_sub(duy, dux), v_sub(sy, sx)), v_sub(my, mx), a5, STRIP_B5, K5);
        if (t.relax_f) {
#pragma unroll
          for (int i = 1; i < 9; ++i) v[i] = v_fma(P.keep_f, fB[i * 32], v[i]);
        }
        // the rest population takes what the others leave of the node's mass: their opposite pairs
        // sum without rounding at the size of u, so the collision keeps the mass that much better
        v[0] = v_sub(drho_p, v_add(v_add(v_add(v[1], v[3]), v_add(v[2], v[4])),
                                   v_add(v_add(v[5], v[7]), v_add(v[6], v[8]))));
        store_row(t.fout, q, v);
        if (EDGE && channel) {  // flux records
          if (inl_a && out_a) S.fi += rho.x * uax.x;
          if (outl_a && out_a) S.fo += rho.x * uax.x;
          if (outl_b && out_b) S.fo += rho.y * uax.y;
        }
      }
    }

    // ===================== phase C: row q2 = r - 2 =====================
    if (THERMAL) {
      const int q2 = r - 2;
      if (q2 >= y0) {
        // central differences of u_act; on a row next to a wall the wall-normal one is the
        // one-sided difference over the two fluid rows; above the pool's top the row repeats
        const bool wlo = !pery && q2 == 0, whi = !pery && !pool && q2 == ny - 1;
        const float2 uyN = (whi || (pool && q2 == ny - 1)) ? uay_p : uay, uyS = wlo ? uay_p : uay_q;
        const float2 divu = v_fma(v_bc(0.5f), dxu_p, v_mul(v_bc((wlo || whi) ? 1.0f : 0.5f), v_sub(uyN, uyS)));
        float2 phi = v_mul(coef_q, divu);
        if (hazi) phi = v_add(phi, hm_q);
        // g collision (Eqs. 16, 18), pairwise as in collide_g
        constexpr float w0 = LatWeights<float>::w0(), w1 = LatWeights<float>::w1(), w5 = LatWeights<float>::w5();
        const float2 T = v_add(P.T_ref, dT_q);
        const float2 xx = v_mul(uax_p, uax_p), yy = v_mul(uay_p, uay_p);
        const float2 Kg = v_fma(P.omega_g, v_fma(v_mul(v_bc(-1.5f), T), v_add(xx, yy), dT_q), phi);
        const float2 K1 = v_mul(v_bc(w1), Kg), K5 = v_mul(v_bc(w5), Kg);
        const float2 wT = v_mul(P.omega_g, T);
        const float2 a1 = v_mul(v_bc(0.5f), wT), a5 = v_mul(v_bc(0.125f), wT);
        const float2 b1 = v_mul(v_bc(STRIP_B1), wT), b5 = v_mul(v_bc(STRIP_B5), wT);
        float2 v[9];
        auto both = [&](int i, int j, float2 cu2, float2 cu, float2 a, float2 b, float2 Kw) {
          const float2 sym = v_fma(a, cu2, Kw), anti = v_mul(b, cu);
          v[i] = v_add(sym, anti);
          v[j] = v_sub(sym, anti);
        };
        v[0] = v_mul(v_bc(w0), Kg);
        both(1, 3, xx, uax_p, a1, b1, K1);
        both(2, 4, yy, uay_p, a1, b1, K1);
        const float2 c5 = v_add(uax_p, uay_p), c6 = v_sub(uay_p, uax_p);
        both(5, 7, v_mul(c5, c5), c5, a5, b5, K5);
        both(6, 8, v_mul(c6, c6), c6, a5, b5, K5);
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = v_fma(P.keep_g, gB[i * 32], v[i]);
        store_row(t.gout, q2, v);
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
    if (hazi) hm_q = hm_p;
    drho_p = drho;
    jx_p = jx;
    jy_p = jy;
    dT_p = dT;
    coef_p = coef;
    if (hazi) hm_p = hm;
    uay_q = uay_p;
    uay_p = uay;
    uax_p = uax;
    dxu_p = dxu;
    psS = psM;
    psM = psN;
  }
  S.bad = !ok;
  // sums of the output nodes only
  if (!out_a) S.m.x = S.e.x = 0.0f;
  if (!out_b) S.m.y = S.e.y = 0.0f;
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
  if constexpr (PCONST) {
    t.nx = I.nx;
    t.ny = I.ny;
    t.pitch = I.pitch;
    t.plane = (int)I.plane;
    t.geometry = I.geometry;
    t.multiphase = I.multiphase;
    t.relax_f = I.omega_f != 1.0;
    t.fin = static_cast<const char*>(par ? I.f[1] : I.f[0]);
    t.gin = static_cast<const char*>(par ? I.g[1] : I.g[0]);
    t.fout = static_cast<char*>(par ? I.f[0] : I.f[1]);
    t.gout = static_cast<char*>(par ? I.g[0] : I.g[1]);
  } else {
    t.nx = uni(I.nx);
    t.ny = uni(I.ny);
    t.pitch = uni(I.pitch);
    t.plane = uni((int)I.plane);
    t.geometry = uni(I.geometry);
    t.multiphase = uni(I.multiphase);
    t.relax_f = uni((int)(I.omega_f != 1.0));
    t.fin = uni(I.f[par]);
    t.gin = uni(I.g[par]);
    t.fout = uni(I.f[par ^ 1]);
    t.gout = uni(I.g[par ^ 1]);
  }
  t.local = uni((int)(ts.step >= 0 ? ts.local : st->local_read != 0));
  t.post_open = uni((int)post_open);
  t.y0 = uni(tile.y0);
  t.y1 = uni(tile.y1);
  const int width = strip_width(cols);
  t.wout = min(width, cols - 8 - w * width);
  t.xs = uni(tile.x0) + w * width - 2;
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
  const double acc[NPART] = {(double)S.m.x + (double)S.m.y, (double)S.e.x + (double)S.e.y, (double)S.h,
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
