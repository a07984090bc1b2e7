"""The records' sums of an FP32 lattice keep the sums' bits.

The first step's record is formed from the initialised populations as they are, so its mass, energy and
heater-row temperature are known: each node's density and temperature deviations are FP32 sums of its
populations in the kernels' order.  The flat launch sums a column's rows four at a time in FP32, from the
bottom of each band, and those sums with the errors carried along (a relative error of about 2^-47 of the
magnitudes summed), and rounds each tile's sums to the fixed-point totals (52 - ceil(log2 m) fraction
bits, m the nodes that feed a total): the totals are exact sums (math.fsum) of the FP32 sums of four rows.
The heater row enters FP64 node by node in every loop.
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


def fours(v, bands):
    """FP32 sums of four rows of a column at a time, from the bottom of each of `bands` bands."""
    ny, out = len(v), []
    start = [b * ny // bands for b in range(bands + 1)]
    for y0, y1 in zip(start, start[1:]):
        for y in range(y0, y1, 4):
            a = v[y]
            for row in v[y + 1:min(y + 4, y1)]:
                a = a + row
            out.append(a)
    assert out[0].dtype == np.float32
    return np.array(out, dtype=np.float64)


# bands: of the flat launch's tiles (13, 6, 13 and 4 rows), None where another kernel runs
@pytest.mark.parametrize("nx,ny,geometry,loop,bands", [
    (1000, 100, "channel", "auto", 8), (599, 80, "walls", "auto", 14), (1500, 150, "channel", "auto", 12),
    (61, 5, "pool", "auto", 2), (1000, 100, "channel", "launches", None), (3000, 300, "walls", "auto", None)])
def test_first_record_is_the_exact_sum(nx, ny, geometry, loop, bands):
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
    assert (lat.step_form == "flat") == (bands is not None)
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
    if bands:
        for got, v, ref in ((d["mass"], drho, rho_ref), (d["energy"], dT, T_ref)):
            sums = fours(v, bands)
            want = math.fsum(sums.ravel()) + n * ref
            assert abs(got - want) <= grid(tiles, n) + 2.0 ** -47 * float(np.abs(sums).sum()) + 1e-15 * n * ref
    heat = math.fsum(dT[0, hx:hx + hl].astype(np.float64))
    T_heat = (p["Tin_R"] + p["dTheat_R"]) * Tc
    want = (T_heat - (heat / hl + T_ref)) / (T_heat - d["energy"] / n)
    # an FP64 sum of the tiles, the totals' grid and the record's own FP64 arithmetic
    assert abs(d["dtstar"] - want) <= (grid(tiles, nx) / hl + 1e-14 * T_heat) / abs(T_heat - d["energy"] / n)
