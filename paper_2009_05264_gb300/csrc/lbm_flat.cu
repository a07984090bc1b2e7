// Kernel instantiations and tile plans of the flat FP32 step.
#include <algorithm>
#include <atomic>
#include <vector>

#include "lbm_flat.cuh"

namespace pplbm {

cudaError_t launch_flat(int thermal, int flags, int warps, const Inst* d_inst, const FlatTile* d_tiles, int ntiles,
                        int grid, int nsteps, FlatState* fstate, unsigned* done, GridBar* bar, unsigned max_polls,
                        cudaStream_t s, const Inst* h_inst) {
  if (ntiles <= 0 || nsteps <= 0) return cudaSuccess;
  if (flat_resident_ctas(thermal, flags, h_inst != nullptr, warps) < 1) return cudaErrorInvalidConfiguration;
  const int insts = h_inst ? 0 : (ntiles + grid - 1) / grid;
  auto go = [&](auto fn) -> cudaError_t {
    // the limit of every launch of this kernel: other threads' lattices share the attribute
    const cudaError_t e = flat_set_smem_limit(fn);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(32 * warps);
    cfg.dynamicSmemBytes = flat_smem_bytes(flags, warps, insts);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    Inst kI{};
    if (h_inst) kI = *h_inst;
    return cudaLaunchKernelEx(&cfg, fn, d_inst, d_tiles, ntiles, nsteps, fstate, done, bar, max_polls,
                              (flags & STEP_RELAX) != 0, kI);
  };
  return thermal ? flat_kernel_for<true>(flags, h_inst != nullptr, go)
                 : flat_kernel_for<false>(flags, h_inst != nullptr, go);
}

// The occupancy calculator's answers are constants of the device: asked once per kernel and CTA size
// (planning asks for all sizes whenever parameters are set).
int flat_resident_ctas(int thermal, int flags, bool single, int warps) {
  constexpr int kDevices = 16;
  static std::atomic<signed char> cache[kDevices][2][4][2][FLAT_MAX_WARPS + 1];  // answer + 1
  int dev = 0;
  if (warps < 1 || warps > FLAT_MAX_WARPS || cudaGetDevice(&dev) != cudaSuccess) return 0;
  std::atomic<signed char>* const known = dev < kDevices ? &cache[dev][thermal != 0][flags & 3][single][warps] : nullptr;
  if (known && known->load() > 0) return known->load() - 1;
  const int insts = single ? 0 : FLAT_MAX_ROUNDS;
  auto get = [&](auto fn) { return flat_resident(fn, flags, warps, insts); };
  const int n = thermal ? flat_kernel_for<true>(flags, single, get) : flat_kernel_for<false>(flags, single, get);
  if (known) known->store((signed char)(n + 1));
  return n;
}

// Strips of an nx-column lattice: as few as 60 columns each allow, of equal even width.
static int flat_strips(int nx) { return (nx + FLAT_WIDTH - 1) / FLAT_WIDTH; }
static int flat_width(int nx) {
  const int ns = flat_strips(nx);
  return ((nx + ns - 1) / ns + 1) / 2 * 2;
}

// Tiles of one instance for bands of at most `rows` rows (of equal height, to a row), appended to
// `out`.  false: a tile has more neighbours than FlatTile holds.
bool build_flat_tiles(int inst, int nx, int ny, int geometry, int rows, std::vector<FlatTile>& out) {
  if (inst >= (1 << 15)) return false;
  const int w = flat_width(nx), ns = (nx + w - 1) / w, nb = (ny + rows - 1) / rows;
  const int base = (int)out.size();
  auto ystart = [&](int b) { return (int)((long long)b * ny / nb); };
  auto band_of = [&](int y) {
    int b = (int)((long long)y * nb / ny);
    while (b > 0 && ystart(b) > y) --b;
    while (b + 1 < nb && ystart(b + 1) <= y) ++b;
    return b;
  };
  const bool perx = geometry != GEOM_CHANNEL, pery = geometry == GEOM_PERIODIC;
  for (int b = 0; b < nb; ++b)
    for (int j = 0; j < ns; ++j) {
      FlatTile t{};
      t.inst = (short)inst;
      t.x0 = j * w;
      t.wout = (short)strip_columns(w, nx - t.x0);
      t.y0 = ystart(b);
      t.rows = ystart(b + 1) - t.y0;
      t.ntiles = ns * nb;
      // the tiles holding what this tile's pulls read: its own rows and columns, 3 around (all of its
      // own rows lie in its band, all of its own columns in its strip)
      std::vector<int> cells;
      const int yhi = t.y0 + t.rows, xhi = std::min(t.x0 + w, nx);
      for (int y : {t.y0 - 3, t.y0 - 2, t.y0 - 1, t.y0, yhi, yhi + 1, yhi + 2}) {
        if (!pery && (y < 0 || y >= ny)) continue;
        const int bb = band_of(((y % ny) + ny) % ny);
        for (int x : {t.x0 - 3, t.x0 - 2, t.x0 - 1, t.x0, xhi, xhi + 1, xhi + 2}) {
          if (!perx && (x < 0 || x >= nx)) continue;
          const int c = base + bb * ns + (((x % nx) + nx) % nx) / w;
          if (c != base + b * ns + j && std::find(cells.begin(), cells.end(), c) == cells.end()) cells.push_back(c);
        }
      }
      if ((int)cells.size() > FLAT_MAX_DEPS) return false;
      t.ndeps = (int)cells.size();
      for (int d = 0; d < t.ndeps; ++d) {
        const int bb = (cells[d] - base) / ns;
        t.deps[d] = cells[d];
        t.dep_rows[d] = (unsigned char)(ystart(bb + 1) - ystart(bb));
      }
      out.push_back(t);
    }
  return true;
}

// Rows per tile for lattices of the given sizes, or 0: the flat kernel does not take them.  Cost
// of a round (every SM running its CTAs' tiles once): a fixed latency chain plus the warps
// that share the SM; fewer rows mean more tiles to spread and less work per SM, but more halo.
// Timed at every height from 4 to 14 on eleven lattices from 100 x 50 to 2500 x 60 (1 to 3 rounds), the
// model picks the fastest one on all of them (1000 x 100: 13 rows 6.71 us a step, 14 rows 6.87, 12
// rows, a second round, 11.2; 600 x 80: 6 rows 5.37, 7 rows 5.49, 5 rows 9.6); so it does with any
// FLAT_ROUND_COST from 0 to 40.
int flat_rows(const std::vector<FlatSize>& sizes, int sms, int max_rounds, const int* per_sm_by_warps) {
  int best = 0;
  double best_cost = 0.0;
  for (int rows = 4; rows <= FLAT_MAX_ROWS; ++rows) {
    long long tiles = 0;
    for (const FlatSize& z : sizes) {
      const int w = flat_width(z.nx);
      tiles += (long long)((z.nx + w - 1) / w) * ((z.ny + rows - 1) / rows);
    }
    const int warps = rows + 6, per_sm = per_sm_by_warps[warps];
    if (per_sm < 1) continue;
    const long long slots = (long long)sms * per_sm;
    const long long rounds = (tiles + slots - 1) / slots;
    if (rounds > max_rounds) continue;
    const long long used = std::min<long long>(per_sm, (tiles + sms - 1) / sms);
    const double cost = (double)rounds * (FLAT_ROUND_COST + (double)(warps * used));
    if (best == 0 || cost < best_cost) {
      best = rows;
      best_cost = cost;
    }
  }
  return best;
}

int flat_max_tiles(int nx, int ny, int sms, int max_rounds) {
  const int w = flat_width(nx), strips = (nx + w - 1) / w;
  long long most = 0;
  for (int rows = 4; rows <= FLAT_MAX_ROWS; ++rows) {
    const long long tiles = (long long)strips * ((ny + rows - 1) / rows);
    const int per_sm = 4 * (16384 / (FLAT_REGS * 32)) / (rows + 6);  // CTAs that the four register files hold
    if (tiles <= (long long)max_rounds * per_sm * sms) most = std::max(most, tiles);
  }
  return (int)most;
}

}  // namespace pplbm
