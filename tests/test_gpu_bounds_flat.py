"""The bounds-checked build on the flat and strip FP32 kernels: wraps, options, several tiles per CTA.

As tests/test_gpu_bounds.py (a child process with the checked library, every global access checked, no
access rejected, the populations those of the default build to rounding), over what its cases leave
out: the flat launch on periodic, walls and pool lattices with last strips of one column, with the bubble
counters, the Hazi-Markus source, tau_f != 1 and isothermal, with more than one tile per CTA and in a
batch of unlike members; the strip kernel's full form, its wraps and its overlapped loop.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

from paper_2009_05264_gb300 import build as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_bounds import ROOT, ROUNDING, fields_for, params_for

STEPS = 25

# name, geometry, nx, ny, overrides, loop, tiling, the form that runs
CASES = [
    ("periodic", "periodic", 61, 33, {"g_a": 0.0}, "auto", None, "flat"),
    ("periodic_tiny", "periodic", 5, 3, {"g_a": 0.0, "tau_f": 0.9}, "auto", None, "flat"),
    ("walls_one_column", "walls", 121, 47, {"tau_f": 0.8, "tau_g": 0.7}, "auto", None, "flat"),
    ("walls_isothermal", "walls", 150, 33, {"thermal": 0}, "auto", None, "flat"),
    ("pool_bubbles", "pool", 121, 64, {"bubble_stats": 1}, "auto", None, "flat"),
    ("channel_hazi", "channel", 131, 40, {"source_model": 1, "tau_f": 1.2}, "auto", None, "flat"),
    ("channel_bubbles_rounds", "channel", 1801, 140, {"bubble_stats": 1}, "auto", None, "flat"),
    ("channel_3x2", "channel", 3, 2, {}, "auto", None, "flat"),
    ("strip_pool_bubbles", "pool", 121, 64, {"bubble_stats": 1}, "launches", None, "strip"),
    ("strip_hazi_barrier", "channel", 131, 40, {"source_model": 1, "tau_f": 1.2}, "persistent", (128, 4), "strip"),
    ("strip_walls_overlapped", "walls", 1681, 180, {}, "persistent", (64, 4), "strip"),
    ("strip_periodic_256", "periodic", 249, 17, {"g_a": 0.0}, "launches", (256, 4), "strip"),
]
BATCH = [("channel", 300, 61, {"bubble_stats": 1}), ("pool", 121, 90, {}), ("periodic", 61, 40, {"g_a": 0.0}),
         ("walls", 500, 77, {"source_model": 1})]


def run_cases(L):
    out = {}
    for k, (name, geometry, nx, ny, extra, loop, tiling, form) in enumerate(CASES):
        p = params_for(geometry, nx, extra)
        lat = L.Lattice(nx, ny, "fp32")
        lat.set_params(p)
        lat.set_step_loop(loop)
        if tiling:
            lat.set_tiling(*tiling)
        assert lat.step_form == form, name
        lat.init_fields(*fields_for(p, nx, ny, 400 + k))
        lat.step(1)
        lat.step(STEPS)
        out[name + ".f"], out[name + ".g"] = lat.populations()
        lat.close()
    b = L.Batch("fp32")
    members = []
    for k, (geometry, nx, ny, extra) in enumerate(BATCH):
        p = params_for(geometry, nx, extra)
        m = b.add(nx, ny, p)
        m.init_fields(*fields_for(p, nx, ny, 500 + k))
        members.append(m)
    assert b.step_form == "flat"
    b.step(STEPS)
    for k, m in enumerate(members):
        out[f"batch{k}.f"], out[f"batch{k}.g"] = m.populations()
    b.close()
    return out


def child_main(lib, out):
    from paper_2009_05264_gb300 import lbm as L

    L.load(path=lib)
    np.savez(out, **run_cases(L))


def test_flat_and_strip_accesses_stay_in_their_buffers(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_05264_gb300 import lbm as L

    lib, out = B.build(bounds_check=True), str(tmp_path / "checked.npz")
    code = (f"import sys; sys.path[:0] = [{ROOT!r}, {os.path.join(ROOT, 'tests')!r}]; import test_gpu_bounds_flat as t; "
            f"t.child_main({lib!r}, {out!r})")
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    got, ref = dict(np.load(out)), run_cases(L)
    assert set(ref) == set(got)
    for key, want in ref.items():
        assert np.abs(got[key] - want).max() <= ROUNDING["fp32"] * np.abs(want).max(), key
