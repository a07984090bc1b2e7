"""FP64 lattices small enough that all tiles are resident: the default tiling's columns and rows.

The tiling only splits the work: the populations of the default tiling agree with those of 128
columns (the plan of larger lattices) to rounding (1e-12 of their scale, the bound between FP64
forms), for widths and heights with ragged last strips and bands, at the smallest heights, and at
tau_f != 1, where the collision keeps part of the pulled populations.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2009_05264_gb300 import inputs as I, params as PP

STEPS = 30


def run(nx, ny, p, fields, tiling):
    from paper_2009_05264_gb300 import lbm as L

    lat = L.Lattice(nx, ny, "fp64")
    lat.set_params(p)
    if tiling is not None:
        lat.set_tiling(*tiling)
    t = lat.tiling
    lat.init_fields(*fields)
    lat.step(STEPS)
    out = lat.populations()
    lat.close()
    return t, out


@pytest.mark.parametrize("nx,ny,geometry,kw", [
    (1000, 100, "channel", {}), (113, 61, "channel", {"tau_f": 0.8}), (57, 4, "channel", {}),
    (40, 3, "channel", {}), (128, 128, "periodic", {"thermal": 0}), (300, 257, "walls", {"tau_f": 1.2}),
    (61, 40, "pool", {}), (400, 30, "channel", {"source_model": 1})])
def test_default_tiling_of_small_lattices(nx, ny, geometry, kw):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    p = PP.resolve(PP.default_params(geometry=geometry, u_in=0.02, dTheat_R=0.05, heat_on_step=5, heater_x0=nx // 3,
                                     heater_len=max(1, nx // 6), g_a=1e-5, **kw), nx)
    fields = I.smooth_random(nx, ny, 5.95, 0.9 * PP.Tc(p), seed=nx + ny, drho=0.002, du=0.004, dT=0.002)
    t, got = run(nx, ny, p, fields, None)
    assert t["cols"] in (64, 128) and t["short_rows"] >= min(4, ny)
    assert run(nx, ny, p, fields, (0, 0))[0] == t  # asked for by name
    t_ref, ref = run(nx, ny, p, fields, (128, 0))
    assert t_ref["cols"] == 128
    for a, b in zip(got, ref):
        if a is not None:
            assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()
