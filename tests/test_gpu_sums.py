"""The records' sums of an FP32 lattice keep the sums' bits.

The first step's record is formed from the initialised populations as they are, so its mass, energy and
heater-row temperature are known: each node's density and temperature deviations are FP32 sums of its
populations in the kernels' order, and their totals are exact sums of those (math.fsum).  The flat launch
sums up to 14 rows of a column in FP32 with the errors carried along (a relative error of about 2^-47 of
the magnitudes summed) and rounds each tile's sums to the fixed-point totals (52 - ceil(log2 m) fraction
bits, m the nodes that feed a total); the heater row enters FP64 node by node in every loop.
"""
import math

import numpy as np
import pytest

import oracle
from paper_2009_05264_gb300 import params as PP

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

W = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]


def grid(tiles, m):
    return tiles * 2.0 ** -(52 - math.ceil(math.log2(m)) + 1)


@pytest.mark.parametrize("nx,ny,geometry,loop", [
    (1000, 100, "channel", "auto"), (599, 80, "walls", "auto"), (1500, 150, "channel", "auto"), (61, 5, "pool", "auto"),
    (1000, 100, "channel", "launches"), (3000, 300, "walls", "auto")])
def test_first_record_is_the_exact_sum(nx, ny, geometry, loop):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_05264_gb300 import lbm as L

    hx, hl = nx // 3 + 1, min(nx // 2, 137)
    p = PP.resolve(PP.default_params(geometry=geometry, u_in=0.02, dTheat_R=0.3, heat_on_step=0, heater_x0=hx,
                                     heater_len=hl, g_a=1e-5), nx)
    rng = np.random.default_rng(nx * ny)
    Tc = oracle.Tc(p)
    rho = 5.95 * (1 + 0.05 * rng.uniform(-1, 1, (ny, nx)))
    T = 0.9 * Tc * (1 + 0.2 * rng.uniform(-1, 1, (ny, nx)))
    lat = L.Lattice(nx, ny, "fp32")
    lat.set_params(p)
    lat.set_step_loop(loop)
    flat = loop == "auto" and nx * ny < 300000
    lat.init_fields(rho, np.zeros_like(rho), np.zeros_like(rho), T)
    f, g = lat.populations()
    rho_ref = p["rho_out"] if geometry == "channel" else p["init_rho_out"]
    T_ref = 0.9 * Tc
    f = (f - W * rho_ref).astype(np.float32)  # the stored deviations
    g = (g - W * T_ref).astype(np.float32)
    drho = ((f[0] + (f[1] + f[3])) + (f[2] + f[4])) + ((f[5] + f[6]) + (f[7] + f[8]))
    dT = (((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7]))) + g[8]
    lat.step(1)
    d = lat.diagnostics()
    n, tiles = nx * ny, -(-nx // 56) * -(-ny // 4)
    if flat:
        mass, energy = (math.fsum(v.astype(np.float64).ravel()) for v in (drho, dT))
        for got, want, ref, v in ((d["mass"], mass, rho_ref, drho), (d["energy"], energy, T_ref, dT)):
            assert abs(got - (want + n * ref)) <= grid(tiles, n) + 2.0 ** -47 * float(np.abs(v).sum()) + 1e-15 * n * ref
    heat = math.fsum(dT[0, hx:hx + hl].astype(np.float64))
    T_heat = (p["Tin_R"] + p["dTheat_R"]) * Tc
    want = (T_heat - (heat / hl + T_ref)) / (T_heat - d["energy"] / n)
    # an FP64 sum of the tiles, the totals' grid and the record's own FP64 arithmetic
    assert abs(d["dtstar"] - want) <= (grid(tiles, nx) / hl + 1e-14 * T_heat) / abs(T_heat - d["energy"] / n)
