"""The FP32 flat launch (a CTA per tile, a warp per row, all steps in one launch) where it can go wrong.

Lattices with the default tiling and few tiles per SM take it.  Sizes around its tile edges (strips
of at most 60 columns of equal even width, bands of at most 15 rows), one tile, tiles of uneven
height, several tiles per CTA, wraps onto the same tile, the first step alone, the full form, the
isothermal step and tau_f != 1: populations and records against one launch per step of the strip
kernel, whose mean density is formed from the same totals (to FP32 rounding, 1e-6 of the population
scale, as for the other loops), and a repeat of the same run bit for bit.  A wait that gives up
ends the launch with LBM_ETIMEOUT and leaves the context usable.
"""
import numpy as np
import pytest

import oracle
from paper_2009_05264_gb300 import inputs as I
from paper_2009_05264_gb300 import params as PP

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROUNDING = 1e-6
STEPS = 50


def lbm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_05264_gb300 import lbm as L

    return L


def case(nx, ny, geometry, **extra):
    base = dict(geometry=geometry, u_in=0.02, dTheat_R=0.1, heat_on_step=5, heater_x0=nx // 3,
                heater_len=max(1, nx // 6), g_a=2e-4)
    base.update(extra)
    p = PP.resolve(PP.default_params(**base), nx)
    return p, I.smooth_random(nx, ny, 5.95, 0.9 * oracle.Tc(p), seed=nx * 5 + ny, drho=0.003, du=0.01, dT=0.003)


def advance(L, nx, ny, p, fields, loop):
    lat = L.Lattice(nx, ny, "fp32")
    lat.set_params(p)
    lat.set_step_loop(loop)
    lat.init_fields(*fields)
    for n in (1, 2, STEPS - 3):
        lat.step(n)
    return lat


@pytest.mark.parametrize("nx,ny,geometry,extra", [
    (3, 2, "channel", {}), (60, 15, "channel", {}), (61, 16, "channel", {}), (121, 31, "channel", {}),
    (179, 61, "channel", {"tau_f": 0.8}), (1300, 200, "channel", {}), (1801, 121, "channel", {}),
    (7, 5, "periodic", {"g_a": 0.0}), (64, 4, "periodic", {"g_a": 0.0}), (251, 90, "periodic", {"g_a": 0.0}),
    (8, 2, "walls", {}), (119, 47, "walls", {}), (150, 33, "walls", {"thermal": 0}),
    (128, 64, "pool", {"bubble_stats": 1}), (333, 29, "channel", {"bubble_stats": 1}),
    (130, 40, "channel", {"source_model": 1, "tau_f": 1.2}),
])
def test_flat_launch_agrees_with_one_launch_per_step(nx, ny, geometry, extra):
    L = lbm()
    p, fields = case(nx, ny, geometry, **extra)
    flat, again, ref = (advance(L, nx, ny, p, fields, loop) for loop in ("auto", "auto", "launches"))
    assert flat.step_loop in ("persistent", "overlapped") and ref.step_loop == "launches"
    assert flat.step_count == ref.step_count == STEPS
    for a, b, c in zip(flat.populations(), again.populations(), ref.populations()):
        assert np.array_equal(a, b)
        assert np.abs(a - c).max() <= ROUNDING * np.abs(c).max()
    rec, rec_ref = flat.diagnostics_range(0, STEPS), ref.diagnostics_range(0, STEPS)
    assert np.array_equal(rec, again.diagnostics_range(0, STEPS))
    assert np.array_equal(rec[:, 0], rec_ref[:, 0])
    for j in range(1, rec.shape[1]):
        if L.DIAG_NAMES[j] == "dp":  # a difference of two pressures: their rounding
            assert np.abs(rec[:, j] - rec_ref[:, j]).max() <= 1e-6
            continue
        scale = max(np.abs(rec_ref[:, j]).max(), 1e-300)
        assert np.abs(rec[:, j] - rec_ref[:, j]).max() <= 100 * ROUNDING * scale, L.DIAG_NAMES[j]


def test_flat_batch_agrees_with_its_members_alone():
    """Members of several sizes and geometries in one flat launch, some CTAs with tiles of two
    members, joining at different steps."""
    L = lbm()
    sizes = [(300, 60, "channel"), (181, 90, "walls"), (128, 128, "pool"), (500, 77, "channel"), (400, 120, "periodic")]
    b = L.Batch("fp32")
    members, cases = [], []
    for nx, ny, geometry in sizes:
        p, fields = case(nx, ny, geometry)
        m = b.add(nx, ny, p)
        m.init_fields(*fields)
        members.append(m)
        cases.append((nx, ny, p, fields))
        b.step(5)
    b.step(20)
    assert b.step_loop in ("persistent", "overlapped")
    for k, (m, (nx, ny, p, fields)) in enumerate(zip(members, cases)):
        steps = 20 + 5 * (len(sizes) - k)
        assert m.step_count == steps
        lat = L.Lattice(nx, ny, "fp32")
        lat.set_params(p)
        lat.set_step_loop("launches")
        lat.init_fields(*fields)
        lat.step(steps)
        for a, c in zip(m.populations(), lat.populations()):
            assert np.abs(a - c).max() <= ROUNDING * np.abs(c).max()
    b.close()


def test_flat_timeout_is_reported_and_the_context_recovers():
    L = lbm()
    nx, ny = 1000, 100
    p, fields = case(nx, ny, "channel")
    lat = L.Lattice(nx, ny, "fp32")
    lat.set_params(p)
    lat.init_fields(*fields)
    assert lat.step_loop == "persistent"
    lat.set_wait_limit(1)
    with pytest.raises(L.LbmError) as err:
        lat.step(20)
    assert err.value.status == 4  # LBM_ETIMEOUT
    lat.set_wait_limit(0)
    lat.init_fields(*fields)
    lat.step(30)
    fresh = L.Lattice(nx, ny, "fp32")
    fresh.set_params(p)
    fresh.init_fields(*fields)
    fresh.step(30)
    for a, b in zip(lat.populations(), fresh.populations()):
        assert np.array_equal(a, b)
