"""The FP32 strip step (a warp per strip of columns, two columns per lane) where it can go wrong.

A strip writes at most 60 columns and pulls 64, in tiles of 56, 120 or 248 columns; strips whose
pulled columns meet an open end, a wrap or the last column take per-lane column offsets.  Widths
around those sizes, odd widths (the last lane's second node outside), one-strip lattices, both
roles of the last strip of a tile, tau_f != 1 (the pulled f kept for the collision), the full
form and the isothermal step, over 60 steps against the FP64 oracle at the FP32 tolerance of the
parity suite (1e-5 of each field's scale).
"""
import numpy as np
import pytest

import oracle
from paper_2009_05264_gb300 import inputs as I
from paper_2009_05264_gb300 import params as PP

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-5
STEPS = 60


@pytest.mark.parametrize("nx,ny,geometry,tiling,extra", [
    *[(nx, 9, "channel", (128, 4), {}) for nx in (5, 58, 60, 62, 63, 65, 119, 121, 124, 185)],
    *[(nx, 8, "walls", (64, 4), {}) for nx in (7, 56, 57, 61, 113)],
    *[(nx, 11, "periodic", (256, 4), {"g_a": 0.0}) for nx in (4, 51, 64, 208, 249, 301)],
    (190, 13, "channel", (256, 5), {}),
    (187, 10, "channel", (128, 0), {"tau_f": 0.8, "tau_g": 0.7}),
    (130, 12, "periodic", (128, 4), {"tau_f": 1.3, "g_a": 0.0}),
    (131, 10, "channel", (128, 4), {"source_model": 1, "tau_f": 0.9}),
    (127, 14, "pool", (128, 5), {"bubble_stats": 1}),
    (150, 9, "walls", (128, 4), {"thermal": 0, "tau_f": 0.9}),
    (150, 9, "channel", (128, 4), {"multiphase": 0}),
])
def test_strip_step_matches_oracle(nx, ny, geometry, tiling, extra):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_05264_gb300 import lbm as L

    base = dict(geometry=geometry, u_in=0.02, dTheat_R=0.1, heat_on_step=5, heater_x0=nx // 3,
                heater_len=max(1, nx // 6), g_a=2e-4)
    base.update(extra)
    p = PP.resolve(PP.default_params(**base), nx)
    fields = I.smooth_random(nx, ny, 5.95, 0.9 * oracle.Tc(p), seed=nx * 7 + ny, drho=0.003, du=0.01, dT=0.003)
    lat = L.Lattice(nx, ny, "fp32")
    lat.set_params(p)
    lat.set_tiling(*tiling)
    lat.init_fields(*fields)
    orc = oracle.Oracle(nx, ny, p)
    orc.init_fields(*fields)
    for n in (1, STEPS - 1):  # one launch, then the loop the library takes
        lat.step(n)
        assert orc.step(n) == 0
    got, ref = lat.fields(), orc.fields()
    u_scale = max(np.abs(ref["ux"]).max(), np.abs(ref["uy"]).max())
    for k in ("rho", "ux", "uy", "T"):
        scale = u_scale if k in ("ux", "uy") else np.abs(ref[k]).max()
        assert np.abs(got[k] - ref[k]).max() < TOL * scale, k
    d, od = lat.diagnostics(), orc.last_diag()
    for k in ("mass", "energy"):
        assert d[k] == pytest.approx(od[k], rel=TOL), k
