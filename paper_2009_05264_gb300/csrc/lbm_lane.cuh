// FP32 arithmetic of one row of a strip: one warp, two adjacent columns per lane.
//
// What the strip kernel (lbm_strip.cuh: a warp marches up its rows) and the flat kernel
// (lbm_flat.cuh: a warp per row) share: pulling a row's populations, the boundary fill, moments,
// equation of state and psi, the force and both collisions of Sec. 2 of Mukherjee, Basu & Mondal
// (arXiv 2009.05264), in packed FP32 (FADD2 / FMUL2 / FFMA2).  Everything but the boundary fill is
// written with explicitly rounded operations, so the results do not depend on the kernel.
//
// Accuracy: the odd part of the f collision takes the momentum and the force themselves, not
// rho u with an approximate 1 / rho, and the rest population closes the node's mass, so the
// velocity error against FP64 is about half the one-column kernel's (3.4e-7 against 1.5e-6 in
// the L2 norm on 1000 x 100 after 500 steps).
#pragma once

#include "lbm_kernels.cuh"

namespace pplbm {

// 3 w of the axis and diagonal links in FP32 (1/3 and 1/12), with 2 B1 + 4 B5 = 1 exactly
constexpr float STRIP_B1 = 0x1.555556p-2f, STRIP_B5 = 0x1.555554p-4f;

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

// psi - psi_ref of one row of the warp: the pair itself, east minus west and east plus west.
struct PsiRow {
  float2 c, d, s;
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

// One lane's view of a strip and the row operations on its two nodes (a: first, b: second).
// EDGE: some pulled column lies outside [1, nx - 2] (an open end, a wrap, or beyond the lattice):
// the links then come from per-lane wrapped columns and the nodes at an open end take the
// boundary fill; otherwise only the wall rows (and a pool's top row) differ from the interior.
// FULL: the pool geometry, the Hazi-Markus source and the bubble statistics.
template <bool THERMAL, bool FULL, bool EDGE>
struct LaneStep {
  const Inst& I;
  const KConst<float>& C;
  const KPair& P;
  const StripTile& t;
  int lane, nx, ny;
  unsigned plane4, pitch4;
  bool perx, pery, channel, pool, multiphase, hazi, bubbles, local;
  int ca, cb;                     // columns of the two nodes (wrapped)
  unsigned oa, ob, om1, op1;      // byte offsets in a row: the nodes, and the columns beside them
  bool inl_a, outl_a, outl_b, out_a, out_b;

  __device__ __forceinline__ LaneStep(const Inst& inst, const StripTile& tile)
      : I(inst), C(inst.strip.C), P(inst.strip.P), t(tile) {
    lane = threadIdx.x & 31;
    nx = t.nx;
    ny = t.ny;
    plane4 = (unsigned)t.plane * 4u;
    pitch4 = (unsigned)t.pitch * 4u;
    perx = t.geometry != GEOM_CHANNEL;
    pery = t.geometry == GEOM_PERIODIC;
    channel = t.geometry == GEOM_CHANNEL;
    pool = FULL && t.geometry == GEOM_POOL;
    multiphase = t.multiphase != 0;
    hazi = FULL && THERMAL && I.source_model == 1;
    bubbles = FULL && I.bubble_stats != 0;
    local = t.local != 0;
    // the strip's halo is two columns a side; lanes beyond it repeat the lane before (unused)
    const int xl = t.xs + 2 * min(lane, t.wout / 2 + 1);
    int cm = xl - 1, cp = xl + 2;
    ca = xl;
    cb = xl + 1;
    if (EDGE) {
      if (perx) {
        ca = wrap_index(xl, nx);
        cb = wrap_index(xl + 1, nx);
        cm = wrap_index(xl - 1, nx);
        cp = wrap_index(xl + 2, nx);
      } else {
        // columns outside the lattice read the end column: never used, and not checked (bad)
        ca = min(max(xl, 0), nx - 1);
        cb = min(max(xl + 1, 0), nx - 1);
        cm = min(max(xl - 1, 0), nx - 1);
        cp = min(max(xl + 2, 0), nx - 1);
      }
    }
    oa = 4u * ca;
    ob = 4u * cb;
    om1 = 4u * cm;
    op1 = 4u * cp;
    inl_a = EDGE && channel && xl == 0;  // xs is even: the inlet column is a lane's first node
    outl_a = EDGE && channel && xl == nx - 1;
    outl_b = EDGE && channel && xl + 1 == nx - 1;
    out_a = lane >= 1 && lane <= t.wout / 2 && xl < nx;
    out_b = out_a && xl + 1 < nx;
  }

  __device__ __forceinline__ bool row_in(int r) const { return pery || (r >= 0 && r < ny); }
  __device__ __forceinline__ int row_of(int r) const { return pery ? wrap_index(r, ny) : r; }

  // bounds-checked builds: `bytes` bytes at p of a population buffer
  __device__ __forceinline__ bool fits(const char* buf, const char* p, int bytes) const {
    return idx_ok(I.st, p - buf, 9LL * t.plane * 4) && idx_ok(I.st, p - buf + bytes - 1, 9LL * t.plane * 4);
  }
  __device__ __forceinline__ float one_at(const char* buf, const char* p) const {
    return fits(buf, p, 4) ? *reinterpret_cast<const float*>(p) : 0.0f;
  }
  // populations of this lane's nodes, shifted by dx columns, of the plane row that starts at p
  __device__ __forceinline__ float2 pair_at(const char* buf, const char* p, int dx) const {
    if (!EDGE) {
      if (dx == 0) return fits(buf, p + oa, 8) ? *reinterpret_cast<const float2*>(p + oa) : make_float2(0.0f, 0.0f);
      return make_float2(one_at(buf, p + oa + 4 * dx), one_at(buf, p + oa + 4 * dx + 4));
    }
    return make_float2(one_at(buf, p + (dx == 0 ? oa : dx < 0 ? om1 : ob)),
                       one_at(buf, p + (dx == 0 ? ob : dx < 0 ? oa : op1)));
  }
  // pulled populations of row r (nothing for rows outside the lattice)
  __device__ __forceinline__ void load_row(int r, float2 (&pf)[9], float2 (&pg)[9]) const {
    if (!row_in(r)) return;
    const int rn = row_of(r);
    const int rm = rn > 0 ? rn - 1 : ny - 1, rp = rn < ny - 1 ? rn + 1 : 0;  // used unless a wall is there
    const size_t n0 = (size_t)(unsigned)rn * pitch4, nm = (size_t)(unsigned)rm * pitch4, np = (size_t)(unsigned)rp * pitch4;
    const bool lo = !pery && rn == 0, hi = !pery && rn == ny - 1;  // hi: a wall, or the pool's top
    if (!local && !lo && !hi) {
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        const size_t o = (size_t)plane4 * i + (lat_cy(i) == 1 ? nm : (lat_cy(i) == -1 ? np : n0));
        pf[i] = pair_at(t.fin, t.fin + o, -lat_cx(i));
        if (THERMAL) pg[i] = pair_at(t.gin, t.gin + o, -lat_cx(i));
        if (EDGE && THERMAL && lat_cx(i) == 1 && inl_a)
          pg[i].x = one_at(t.gin, t.gin + (size_t)plane4 * lat_opp(i) + n0 + oa);
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
          if (EDGE && THERMAL && lat_cx(i) == 1 && inl_a)
            pg[i].x = one_at(t.gin, t.gin + (size_t)plane4 * lat_opp(i) + n0 + oa);
        }
      }
    }
  }
  // stores of the nine populations of row y
  __device__ __forceinline__ void store_row(char* buf, int y, const float2 (&v)[9]) const {
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
  }

  // Boundary nodes of lattice row rn: the wall rows' temperatures (a link from a wall holds the
  // node's own opposite population, see load_row), the open ends, the pool's top row.  The closed
  // forms are boundary_fill's; the populations that it reads again from memory are at hand here: an
  // inlet node's opposite g in place of its unknown links, and an outlet node's g in the lane of
  // the node before it.
  __device__ __forceinline__ void fill(int rn, long long step, float2 (&pf)[9], float2 (&pg)[9]) const {
    if (local) return;
    const bool lo = !pery && rn == 0, hi = !pery && !pool && rn == ny - 1;
    if (THERMAL && (lo || hi)) {
      const bool heat_bc = I.heater_len > 0 && (step - 1) >= I.heat_on_step;
      auto wall_T = [&](int xn, int i) {
        if (lat_cy(i) != 1 || !heat_bc) return C.dT_in;
        int sx = xn - lat_cx(i);
        if (perx) sx = sx < 0 ? sx + nx : (sx >= nx ? sx - nx : sx);
        return sx >= I.heater_x0 && sx < I.heater_x0 + I.heater_len ? C.dT_heat : C.dT_in;
      };
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        if ((lat_cy(i) == 1 && lo) || (lat_cy(i) == -1 && hi)) {
          const float2 Tw = make_float2(wall_T(ca, i), wall_T(cb, i));
          pg[i] = v_sub(v_mul(v_bc(2.0f * lat_w<float>(i)), Tw), pg[i]);
        }
      }
    }
    if constexpr (EDGE) {
      if (channel) {
        if (inl_a) {
          open_end(pf, 0, NodeBC{lo, hi, true, false, false});
          if (THERMAL) {
            // anti-bounce-back at the inlet temperature
#pragma unroll
            for (int i = 0; i < 9; ++i)
              if (lat_cx(i) == 1 && !(lat_cy(i) == 1 && lo) && !(lat_cy(i) == -1 && hi))
                pg[i].x = __fmaf_rn(2.0f * lat_w<float>(i), C.dT_in, -pg[i].x);
          }
        }
        if (outl_a) {
          open_end(pf, 0, NodeBC{lo, hi, false, true, false});
          // the lane's second column is outside: a copy, so that it is outside the EOS domain only with the node
#pragma unroll
          for (int i = 0; i < 9; ++i) pf[i].y = pf[i].x;
        }
        if (outl_b) open_end(pf, 1, NodeBC{lo, hi, false, true, false});
        if (THERMAL && t.xs + t.wout + 3 >= nx - 1) {
          // zero temperature gradient: all nine populations of node nx - 2, wall links included
#pragma unroll
          for (int i = 0; i < 9; ++i) {
            const float before = __shfl_up_sync(0xffffffffu, pg[i].y, 1);
            if (outl_a) pg[i].x = pg[i].y = before;
            if (outl_b) pg[i].y = pg[i].x;
          }
        }
      }
    }
    if constexpr (FULL) {
      if (pool && rn == ny - 1) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int xn = h ? cb : ca;
          float f1[9], g1[9];
#pragma unroll
          for (int i = 0; i < 9; ++i) {
            f1[i] = h ? pf[i].y : pf[i].x;
            g1[i] = h ? pg[i].y : pg[i].x;
          }
          boundary_fill<float, THERMAL>(f1, g1, NodeBC{false, false, false, false, true}, I, C,
                                        reinterpret_cast<const float*>(t.gin), t.plane, t.pitch, rn * t.pitch + xn, xn,
                                        perx, step);
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
  }
  // Zou-He conditions of one node (h: which of the lane's) at an open end: f only.
  __device__ __forceinline__ void open_end(float2 (&pf)[9], int h, const NodeBC& nb) const {
    float f1[9], g1[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) f1[i] = h ? pf[i].y : pf[i].x;
    boundary_fill<float, false>(f1, g1, nb, I, C, nullptr, 0, 0, 0, 0, false, 0);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      if (h) pf[i].y = f1[i];
      else pf[i].x = f1[i];
    }
  }

  // Mass that row rn's pull took in minus the mass it let out through the open ends (this lane's
  // output nodes): in, the open-end links that the boundary fill set; out, the node's
  // post-collision populations that point out of the open end (no node pulls them; at a wall row
  // the diagonal one is bounced back instead).
  __device__ __forceinline__ double open_mass(int rn, const float2 (&pf)[9]) const {
    double sum = 0.0;
    const bool lo = rn == 0, hi = rn == ny - 1;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const bool inl = h == 0 && inl_a, outl = h ? outl_b : outl_a;
      if (!(h ? out_b : out_a)) continue;
      const char* const pn = t.fin + (size_t)rn * pitch4 + (h ? ob : oa);
      auto fl = [&](int i) { return (double)one_at(t.fin, pn + (size_t)plane4 * i); };
      auto fc = [&](int i) { return (double)(h ? pf[i].y : pf[i].x); };
      if (inl)
        sum += fc(1) + (lo ? 0.0 : fc(5)) + (hi ? 0.0 : fc(8)) - (fl(3) + (hi ? 0.0 : fl(6)) + (lo ? 0.0 : fl(7)));
      else if (outl)
        sum += fc(3) + (lo ? 0.0 : fc(6)) + (hi ? 0.0 : fc(7)) - (fl(1) + (hi ? 0.0 : fl(5)) + (lo ? 0.0 : fl(8)));
    }
    return sum;
  }

  // Moments (Eqs. 4, 6, 17), equation of state (Eq. 12), psi (Eq. 11) and the factor of the energy
  // source (Eq. 19) of a row.  ok: cleared where a node is outside the EOS domain.
  struct Node {
    float2 drho, jx, jy, dT, coef, hm, dpsi, drad;  // hm: first Eq. 19, T (dp/dT)_rho / (rho^2 c_v)
  };
  __device__ __forceinline__ void node(const float2 (&pf)[9], const float2 (&pg)[9], Node& n, bool& ok) const {
    const float2 zero = make_float2(0.0f, 0.0f);
    const float2 p56 = v_add(pf[5], pf[6]), p78 = v_add(pf[7], pf[8]);
    n.drho = v_add(v_add(v_add(pf[0], v_add(pf[1], pf[3])), v_add(pf[2], pf[4])), v_add(p56, p78));
    n.jx = v_add(v_sub(pf[1], pf[3]), v_add(v_sub(pf[5], pf[6]), v_sub(pf[8], pf[7])));
    n.jy = v_add(v_sub(pf[2], pf[4]), v_sub(p56, p78));
    const float2 rho = v_add(P.rho_ref, n.drho);
    float2 T = P.T0;
    if (THERMAL) {
      n.dT = v_add(v_add(v_add(v_add(pg[0], pg[1]), v_add(pg[2], pg[3])),
                         v_add(v_add(pg[4], pg[5]), v_add(pg[6], pg[7]))), pg[8]);
      T = v_add(P.T_ref, n.dT);
    }
    n.drad = n.dpsi = zero;
    ok = ok && rho.x > 0.0f && rho.y > 0.0f;
    if (multiphase) {
      // exact differences from the reference state; with om = 1 - b rho,
      // D = 1 + 2 b rho - (b rho)^2 = 2 - om^2
      const float2 nv = v_fma(P.b, rho, v_bc(-1.0f));
      const float2 om = v_mul(nv, v_bc(-1.0f));
      const float2 invD = v_rcp(v_fma(nv, om, v_bc(2.0f)));
      const float2 inv1 = v_rcp(om);
      float2 z = v_mul(n.drho, v_mul(v_fma(P.s3, rho, P.rho_ref), invD));
      float2 sa = zero, isT = zero, drad = v_mul(v_mul(n.drho, T), inv1);
      if (THERMAL) {
        // sqrt(alpha) relative to its reference value: 1 + m1 (sqrt T - sqrt T_ref), the
        // difference of the roots as dT / (sqrt T + sqrt T_ref)
        isT = v_rsqrt(T);
        const float2 w = v_mul(n.dT, v_rcp(v_fma(T, isT, P.sqrtT_r)));
        sa = v_fma(P.m1, w, v_bc(1.0f));
        z = v_mul(v_mul(sa, sa), z);
        drad = v_mul(P.cA, v_fma(P.rho_ref, n.dT, drad));
        drad = v_fma(P.cB, z, drad);
        drad = v_fma(P.cK, v_mul(w, v_add(sa, v_bc(1.0f))), drad);
      } else {
        drad = v_fma(P.cB, z, v_mul(P.cA, drad));
      }
      drad = v_fma(P.c3, n.drho, drad);
      const float2 rad = v_add(P.rad_ref, drad);
      const float2 psi = make_float2(s_sqrt(fmaxf(rad.x, 0.0f)), s_sqrt(fmaxf(rad.y, 0.0f)));
      const float2 den = v_add(psi, P.psi_ref);  // zero only where drad is
      n.drad = drad;
      n.dpsi = v_mul(drad, v_rcp(make_float2(fmaxf(den.x, 1e-30f), fmaxf(den.y, 1e-30f))));
      ok = ok && om.x > 0.0f && om.y > 0.0f && rad.x >= 0.0f && rad.y >= 0.0f;
      if (THERMAL) {  // T (1 - (dp/dT)_rho / (rho c_v)) of the second Eq. 19
        const float2 q = v_mul(v_mul(sa, isT), v_mul(rho, invD));
        const float2 Te = v_mul(T, v_fma(P.cR, inv1, v_mul(P.cS, q)));
        n.coef = v_sub(T, Te);
        if (hazi) {  // first Eq. 19
          n.coef = T;
          n.hm = v_mul(Te, v_rcp(rho));
        }
      }
    } else if (THERMAL) {
      n.coef = T;
      ok = ok && fabsf(T.x) < INFINITY && fabsf(T.y) < INFINITY;
    }
  }

  // Whether a node of the lattice was outside the EOS domain (ok: what node left of it over the lane's
  // rows).  A lane with both columns beyond an open end holds none.
  __device__ __forceinline__ bool bad(bool ok) const {
    const int xl = t.xs + 2 * lane;
    return !ok && !(EDGE && channel && (xl < 0 || xl >= nx));
  }

  // Hazi-Markus: the source's density-gradient term of this lane's output nodes of lattice row rn,
  // with rho^n - rho^(n-1) as deviations from rho_ref; the lane owns the nodes' history (read,
  // then overwritten with rho^n).
  __device__ __forceinline__ void history(int rn, Node& n) const {
    float* const rho_prev = static_cast<float*>(I.rho_prev);
    const int k = rn * t.pitch + ca;
    if (out_a && idx_ok(I.st, k, t.plane)) {
      n.hm.x = n.hm.x * (n.drho.x - rho_prev[k]);
      rho_prev[k] = n.drho.x;
    }
    if (out_b && idx_ok(I.st, k + 1, t.plane)) {
      n.hm.y = n.hm.y * (n.drho.y - rho_prev[k + 1]);
      rho_prev[k + 1] = n.drho.y;
    }
  }
  // Pressure probes at (1, ny / 2) and (nx - 2, ny / 2) of a channel: put(0 or 1, pressure).
  template <typename Put>
  __device__ __forceinline__ void probes(int rn, const Node& n, const Put& put) const {
    if constexpr (!EDGE) return;
    if (!channel || rn != ny / 2) return;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int xn = h ? cb : ca;
      if ((h ? out_b : out_a) && (xn == 1 || xn == nx - 2)) {
        const float dr = h ? n.drho.y : n.drho.x;
        const float p = multiphase ? P.p_ref + ((h ? n.drad.y : n.drad.x) * P.inv_ps + dr * (1.0f / 3.0f))
                                   : ((h ? P.rho_ref.y : P.rho_ref.x) + dr) * (1.0f / 3.0f);
        if (xn == 1) put(0, p);
        if (xn == nx - 2) put(1, p);
      }
    }
  }
  // Heater-row temperatures of this lane's output nodes of row 0 (zero beside the heater).
  __device__ __forceinline__ float2 heater_dT(const float2& dT) const {
    return make_float2(out_a && ca >= I.heater_x0 && ca < I.heater_x0 + I.heater_len ? dT.x : 0.0f,
                       out_b && cb >= I.heater_x0 && cb < I.heater_x0 + I.heater_len ? dT.y : 0.0f);
  }

  // East and west neighbours of a row's values, from the adjacent lanes; at the open ends the
  // ghost column repeats the end column.
  __device__ __forceinline__ void east_west(const float2& v, float2& E, float2& W) const {
    float w = __shfl_up_sync(0xffffffffu, v.y, 1), e = __shfl_down_sync(0xffffffffu, v.x, 1);
    float ea = v.y;
    if (EDGE) {
      if (inl_a) w = v.x;
      if (outl_a) ea = v.x;
      if (outl_b) e = v.y;
    }
    E = make_float2(ea, e);
    W = make_float2(w, v.x);
  }
  __device__ __forceinline__ PsiRow psi_row(const float2& dpsi) const {
    float2 E, W;
    east_west(dpsi, E, W);
    return PsiRow{dpsi, v_sub(E, W), v_add(E, W)};
  }

  // Force (Eqs. 9, 10, 14, 15) and velocities (Eqs. 6, 7) of row q from psi of the rows around it.
  struct Flow {
    float2 Fx, Fy, rho, ux, uy, dux, duy, uax, uay;
  };
  __device__ __forceinline__ Flow flow(int q, const PsiRow& N, const PsiRow& M, const PsiRow& S, const float2& drho,
                                       const float2& jx, const float2& jy, float rra) const {
    Flow o;
    o.Fx = o.Fy = make_float2(0.0f, 0.0f);
    if (multiphase) {
      // t1 = sum G_i d_i c_i, t2 = sum G_i d_i^2 c_i of d = psi - psi_ref, the squares as products
      // of sums and differences; the diagonal part of t2y is
      // Gh (E_N^2 + W_N^2 - E_S^2 - W_S^2) = Gh / 2 [(s_N - s_S)(s_N + s_S) + (d_N - d_S)(d_N + d_S)]
      const float2 dsum = v_add(N.d, S.d);
      const float2 gd = v_mul(P.G2, M.d);
      const float2 t1x = v_fma(P.Gh, dsum, gd);
      const float2 cdif = v_sub(N.c, S.c), sdif = v_sub(N.s, S.s);
      const float2 gc = v_mul(P.G2, cdif);
      const float2 t1y = v_fma(P.Gh, sdif, gc);
      const float2 t2x = v_fma(gd, M.s, v_mul(P.Gh, v_fma(N.d, N.s, v_mul(S.d, S.s))));
      const float2 m = v_fma(sdif, v_add(N.s, S.s), v_mul(v_sub(N.d, S.d), dsum));
      const float2 t2y = v_fma(gc, v_add(N.c, S.c), v_mul(P.Ghh, m));
      const float2 nlead = v_fma(P.nbeta, M.c, P.npsi_ref);
      o.Fx = v_fma(nlead, t1x, v_mul(P.nmix, t2x));
      o.Fy = v_fma(nlead, t1y, v_mul(P.nmix, t2y));
      if (!pery && q == 0) o.Fy = v_add(o.Fy, v_fma(M.c, P.wall1, P.wall0));
      if (!pery && !pool && q == ny - 1) o.Fy = v_sub(o.Fy, v_fma(M.c, P.wall1, P.wall0));
    }
    o.Fy = v_fma(v_add(drho, v_bc(rra)), P.ng_a, o.Fy);  // Eq. 14, gravity along -y
    o.rho = v_add(P.rho_ref, drho);
    const float2 irho = v_rcp(o.rho);
    o.ux = v_mul(jx, irho);
    o.uy = v_mul(jy, irho);
    o.dux = v_mul(o.Fx, irho);
    o.duy = v_mul(o.Fy, irho);
    o.uax = v_fma(v_bc(0.5f), o.dux, o.ux);  // Eq. 7
    o.uay = v_fma(v_bc(0.5f), o.duy, o.uy);
    return o;
  }

  // f collision (Eqs. 2, 3, 5), pairwise over opposite directions as in collide_f.  The odd
  // part, 3 w c.(omega rho u + rho du), takes the momentum and the force themselves: the
  // error of the approximate 1 / rho in u would act on the momentum every step.  B1 and B5
  // keep 2 B1 + 4 B5 = 1, and 4.5 w of the axis and diagonal links are exact.  old(i): the
  // pulled population i, asked for only when tau_f != 1.
  template <typename Old>
  __device__ __forceinline__ void collide_f(const Flow& o, const float2& drho, const float2& jx, const float2& jy,
                                            const Old& old, float2 (&v)[9]) const {
    constexpr float w1 = LatWeights<float>::w1(), w5 = LatWeights<float>::w5();
    const float2 sx = v_fma(v_bc(2.0f), o.ux, o.dux), sy = v_fma(v_bc(2.0f), o.uy, o.duy);
    const float2 dsx = v_mul(o.dux, sx), dsy = v_mul(o.duy, sy);
    const float2 usq = v_fma(o.ux, o.ux, v_mul(o.uy, o.uy));
    const float2 nr15 = v_mul(v_bc(-1.5f), o.rho);
    const float2 K = v_fma(nr15, v_add(dsx, dsy), v_mul(P.omega_f, v_fma(nr15, usq, drho)));
    const float2 K1 = v_mul(v_bc(w1), K), K5 = v_mul(v_bc(w5), K);
    const float2 a1 = v_mul(v_bc(0.5f), o.rho), a5 = v_mul(v_bc(0.125f), o.rho);
    const float2 mx = v_fma(P.omega_f, jx, o.Fx), my = v_fma(P.omega_f, jy, o.Fy);
    auto both = [&](int i, int j, float2 cu, float2 cds, float2 m, float2 a, float b, float2 Kw) {
      const float2 sym = v_fma(a, v_fma(v_mul(P.omega_f, cu), cu, cds), Kw), anti = v_mul(v_bc(b), m);
      v[i] = v_add(sym, anti);
      v[j] = v_sub(sym, anti);
    };
    both(1, 3, o.ux, dsx, mx, a1, STRIP_B1, K1);
    both(2, 4, o.uy, dsy, my, a1, STRIP_B1, K1);
    both(5, 7, v_add(o.ux, o.uy), v_mul(v_add(o.dux, o.duy), v_add(sx, sy)), v_add(mx, my), a5, STRIP_B5, K5);
    both(6, 8, v_sub(o.uy, o.ux), v_mul(v_sub(o.duy, o.dux), v_sub(sy, sx)), v_sub(my, mx), a5, STRIP_B5, K5);
    if (t.relax_f) {
#pragma unroll
      for (int i = 1; i < 9; ++i) v[i] = v_fma(P.keep_f, old(i), v[i]);
    }
    // the rest population takes what the others leave of the node's mass: their opposite pairs
    // sum without rounding at the size of u, so the collision keeps the mass that much better
    v[0] = v_sub(drho, v_add(v_add(v_add(v[1], v[3]), v_add(v[2], v[4])),
                             v_add(v_add(v[5], v[7]), v_add(v[6], v[8]))));
  }

  // Source and g collision (Eqs. 16, 18, 19) of row q2, pairwise as in collide_g: u_act of the row
  // (uax, uay) and of the rows above and below (uyN, uyS), dxu its u_x east minus west.  Central
  // differences; on a row next to a wall the wall-normal one is the one-sided difference over the
  // two fluid rows; above the pool's top the row repeats.
  template <typename Old>
  __device__ __forceinline__ void collide_g(int q2, const float2& uax, const float2& uay, const float2& uyN,
                                            const float2& uyS, const float2& dxu, const float2& dT, const float2& coef,
                                            const float2& hm, const Old& old, float2 (&v)[9]) const {
    constexpr float w0 = LatWeights<float>::w0(), w1 = LatWeights<float>::w1(), w5 = LatWeights<float>::w5();
    const bool wlo = !pery && q2 == 0, whi = !pery && !pool && q2 == ny - 1;
    const float2 n = (whi || (pool && q2 == ny - 1)) ? uay : uyN, s = wlo ? uay : uyS;
    const float2 divu = v_fma(v_bc(0.5f), dxu, v_mul(v_bc((wlo || whi) ? 1.0f : 0.5f), v_sub(n, s)));
    float2 phi = v_mul(coef, divu);
    if (hazi) phi = v_add(phi, hm);
    const float2 T = v_add(P.T_ref, dT);
    const float2 xx = v_mul(uax, uax), yy = v_mul(uay, uay);
    const float2 Kg = v_fma(P.omega_g, v_fma(v_mul(v_bc(-1.5f), T), v_add(xx, yy), dT), phi);
    const float2 K1 = v_mul(v_bc(w1), Kg), K5 = v_mul(v_bc(w5), Kg);
    const float2 wT = v_mul(P.omega_g, T);
    const float2 a1 = v_mul(v_bc(0.5f), wT), a5 = v_mul(v_bc(0.125f), wT);
    const float2 b1 = v_mul(v_bc(STRIP_B1), wT), b5 = v_mul(v_bc(STRIP_B5), wT);
    auto both = [&](int i, int j, float2 cu2, float2 cu, float2 a, float2 b, float2 Kw) {
      const float2 sym = v_fma(a, cu2, Kw), anti = v_mul(b, cu);
      v[i] = v_add(sym, anti);
      v[j] = v_sub(sym, anti);
    };
    v[0] = v_mul(v_bc(w0), Kg);
    both(1, 3, xx, uax, a1, b1, K1);
    both(2, 4, yy, uay, a1, b1, K1);
    const float2 c5 = v_add(uax, uay), c6 = v_sub(uay, uax);
    both(5, 7, v_mul(c5, c5), c5, a5, b5, K5);
    both(6, 8, v_mul(c6, c6), c6, a5, b5, K5);
#pragma unroll
    for (int i = 0; i < 9; ++i) v[i] = v_fma(P.keep_g, old(i), v[i]);
  }
};

// A strip's uniform description for one step: everything of the lattice and of the step's buffers
// (par: the parity of the step); the columns and rows are the caller's to set.
template <bool PCONST>
__device__ __forceinline__ void strip_tile_consts(StripTile& t, const Inst& I, int par, bool local, bool post_open) {
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
  t.local = uni((int)local);
  t.post_open = uni((int)post_open);
}

}  // namespace pplbm
