"""Waits of the flat launch that give up at any point of it end the launch and leave the context usable.

Poll limits from one poll up make waits run out in the first steps or far into the launch, in warps of
either kind, with one tile per CTA, with several, and in a batch: the call reports LBM_ETIMEOUT or, if
every wait was shorter, succeeds; after a new initialisation the lattice steps as a fresh one, bit for
bit.  (That all warps of a CTA see the same decision in the same turn is by construction.)
"""
import numpy as np
import pytest

from paper_2009_05264_gb300 import inputs as I
from paper_2009_05264_gb300 import params as PP

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LIMITS = (1, 2, 5, 10, 20, 50)
TIMEOUT = 4  # LBM_ETIMEOUT


def case(nx, ny, geometry="channel"):
    p = PP.resolve(PP.default_params(geometry=geometry, u_in=0.02, dTheat_R=0.05, heat_on_step=5, heater_x0=nx // 3,
                                     heater_len=20, g_a=1e-5), nx)
    return p, I.smooth_random(nx, ny, 5.95, 0.9 * PP.Tc(p), seed=nx + ny, drho=0.002, du=0.004, dT=0.002)


def tolerated(step):
    from paper_2009_05264_gb300 import lbm as L

    try:
        step()
    except L.LbmError as e:
        assert e.status == TIMEOUT


@pytest.mark.parametrize("nx,ny,loop", [(600, 80, "persistent"), (1500, 150, "overlapped")])
def test_lattice(nx, ny, loop):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_05264_gb300 import lbm as L

    p, fields = case(nx, ny)
    lat, fresh = L.Lattice(nx, ny, "fp32"), L.Lattice(nx, ny, "fp32")
    for a in (lat, fresh):
        a.set_params(p)
    assert lat.step_loop == loop
    for limit in LIMITS:
        lat.set_wait_limit(limit)
        lat.init_fields(*fields)
        tolerated(lambda: lat.step(40))
    lat.set_wait_limit(0)
    for a in (lat, fresh):
        a.init_fields(*fields)
        a.step(30)
    for x, y in zip(lat.populations(), fresh.populations()):
        assert np.array_equal(x, y)


def test_batch():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_05264_gb300 import lbm as L

    cases = [(nx, ny, *case(nx, ny, g)) for nx, ny, g in ((300, 90, "channel"), (128, 400, "pool"), (500, 250, "walls"))]
    b, fresh = L.Batch("fp32"), L.Batch("fp32")
    members = [[x.add(nx, ny, p) for nx, ny, p, _ in cases] for x in (b, fresh)]
    assert b.step_loop in ("persistent", "overlapped")

    def start(ms):
        for m, (_, _, _, fields) in zip(ms, cases):
            m.init_fields(*fields)

    for limit in LIMITS:
        b.set_wait_limit(limit)
        start(members[0])
        tolerated(lambda: b.step(40))
    b.set_wait_limit(0)
    for x, ms in zip((b, fresh), members):
        start(ms)
        x.step(30)
    for m, r in zip(*members):
        for x, y in zip(m.populations(), r.populations()):
            assert np.array_equal(x, y)
