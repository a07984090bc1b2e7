"""Lattices that wrap in x and end in a strip or tile of one or two columns.

The lanes (or threads) past the last column wrap to the first columns of the lattice.  They must pull
only columns that the tile waits for: a node formed from populations of another step, or from the
fields that init_fields and fields() stage in the spare buffer, would report a healthy lattice as
unstable.  Repeated segments of initialisation, a few steps and a readback, in the flat launch, in the
FP32 strip kernel's and in the FP64 kernel's overlapped loop: no error, and the populations of one
launch per step to rounding (1e-6 and 1e-12 of their scale, the bounds between loops elsewhere).
"""
import numpy as np
import pytest

from paper_2009_05264_gb300 import inputs as I
from paper_2009_05264_gb300 import params as PP

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROUNDING = {"fp64": 1e-12, "fp32": 1e-6}


@pytest.mark.parametrize("nx,ny,geometry,prec,tiling,loop", [
    *[(nx, 60, g, "fp32", None, "auto") for nx in (1741, 1742, 1801) for g in ("walls", "periodic", "pool")],
    *[(nx, 180, g, p, (64, 4), "persistent") for nx in (1681, 1682) for g, p in (("walls", "fp32"), ("periodic", "fp32"),
                                                                                ("walls", "fp64"))],
])
def test_last_columns_of_a_wrap(nx, ny, geometry, prec, tiling, loop):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_05264_gb300 import lbm as L

    p = PP.resolve(PP.default_params(geometry=geometry, u_in=0.0, dTheat_R=0.1, heat_on_step=5, heater_x0=nx // 3,
                                     heater_len=40, g_a=0.0 if geometry == "periodic" else 2e-4), nx)
    fields = I.smooth_random(nx, ny, 5.95, 0.9 * PP.Tc(p), seed=nx + ny, drho=0.003, du=0.01, dT=0.003)

    def lattice(loop):
        lat = L.Lattice(nx, ny, prec)
        lat.set_params(p)
        lat.set_step_loop(loop)
        if tiling:
            lat.set_tiling(*tiling)
        return lat

    lat, ref = lattice(loop), lattice("launches")
    assert lat.step_loop == "overlapped" if tiling else lat.step_loop in ("persistent", "overlapped")
    for _ in range(10):
        lat.init_fields(*fields)
        for n in (2, 3, 10):
            lat.step(n)
            lat.fields()
    ref.init_fields(*fields)
    ref.step(15)
    for a, b in zip(lat.populations(), ref.populations()):
        assert np.abs(a - b).max() <= ROUNDING[prec] * np.abs(b).max()
