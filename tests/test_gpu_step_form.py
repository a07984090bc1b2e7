"""The kernel that runs, by name, and every FP32 kernel and loop against each other.

step_form names the kernel of a multi-step call: it follows the kernel and loop requests, the precision,
the options and the tiling.  One lattice then goes through each FP32 kernel and loop, each named so that
no two entries are the same launch: they agree with the one-column kernel to 1e-5 of the populations'
scale after 60 steps (two different orders of the collision's roundings, as the other form tests allow),
and the strip and flat kernels, which share their arithmetic, with each other to 1e-6 (the mean density's
rounding, as between loops elsewhere).
"""
import numpy as np
import pytest

from paper_2009_05264_gb300 import inputs as I
from paper_2009_05264_gb300 import params as PP

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def lbm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_05264_gb300 import lbm as L

    return L


def prm(nx, **extra):
    base = dict(geometry="channel", u_in=0.02, dTheat_R=0.05, heat_on_step=5, heater_x0=nx // 3, heater_len=20, g_a=1e-5)
    base.update(extra)
    return PP.resolve(PP.default_params(**base), nx)


def test_form_of_a_lattice():
    L = lbm()
    lat = L.Lattice(260, 41, "fp32")
    lat.set_params(prm(260))
    assert lat.step_form == "flat"
    for extra in ({"bubble_stats": 1}, {"source_model": 1}, {"thermal": 0}, {"geometry": "pool"}):
        lat.set_params(prm(260, **extra))
        assert lat.step_form == "flat"  # whatever the form asked for is called
    lat.set_params(prm(260))
    lat.set_step_loop("launches")
    assert lat.step_form == "strip"
    lat.set_step_loop("auto")
    for kernel, form in (("scalar", "scalar"), ("tma", "tma"), ("paired", "flat"), ("interior", "flat"), ("auto", "flat")):
        lat.set_kernel(kernel)
        assert lat.step_form == form
    lat.set_tiling(128, 8)
    assert lat.step_form == "strip"
    lat.set_tiling(0, 0)
    assert lat.step_form == "flat"
    big, f64 = L.Lattice(4000, 400, "fp32"), L.Lattice(260, 41, "fp64")
    for a, form in ((big, "strip"), (f64, "interior")):
        a.set_params(prm(a.nx))
        assert a.step_form == form
    f64.set_params(prm(260, bubble_stats=1))
    assert f64.step_form == "scalar"


def test_form_of_a_batch():
    L = lbm()
    b = L.Batch("fp32")
    for nx, ny in ((150, 40), (333, 61)):
        b.add(nx, ny, prm(nx))
    assert b.step_form == "flat"
    b.set_step_loop("launches")
    assert b.step_form == "strip"
    b.set_kernel("scalar")
    assert b.step_form == "scalar"
    b.close()


def test_every_fp32_kernel_and_loop_agrees():
    L = lbm()
    nx, ny = 1800, 160
    p = prm(nx)
    fields = I.smooth_random(nx, ny, 5.95, 0.9 * PP.Tc(p), seed=11, drho=0.002, du=0.005, dT=0.002)
    pops = {}
    for kernel, loop, tiling, form, runs in (
            ("scalar", "launches", (128, 16), "scalar", "launches"), ("tma", "launches", (128, 16), "tma", "launches"),
            ("auto", "launches", (128, 16), "strip", "launches"), ("auto", "persistent", (128, 16), "strip", "persistent"),
            ("auto", "persistent", (64, 4), "strip", "overlapped"), ("auto", "auto", (0, 0), "flat", "overlapped")):
        lat = L.Lattice(nx, ny, "fp32")
        lat.set_params(p)
        lat.set_kernel(kernel)
        lat.set_step_loop(loop)
        lat.set_tiling(*tiling)
        assert (lat.step_form, lat.step_loop) == (form, runs)
        lat.init_fields(*fields)
        lat.step(60)
        pops[form, runs] = lat.populations()
        lat.close()
    assert len(pops) == 6
    for key, got in pops.items():
        for a, b in zip(got, pops["scalar", "launches"]):
            assert np.abs(a - b).max() < 1e-5 * np.abs(b).max(), key
        if key[0] in ("strip", "flat"):
            for a, b in zip(got, pops["strip", "launches"]):
                assert np.abs(a - b).max() <= 1e-6 * np.abs(b).max(), key
