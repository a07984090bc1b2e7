"""Lattices stepped from several host threads at once, each thread with its own.

The flat launch's dynamic shared memory depends on the rows of a tile and on tau_f, and lattices of
different sizes share a kernel: no thread's launch may be refused because of another's, and every
lattice ends as it does alone, bit for bit.
"""
import threading

import numpy as np
import pytest

from paper_2009_05264_gb300 import inputs as I
from paper_2009_05264_gb300 import params as PP

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CALLS = 4000
SIZES = [(1000, 100, {}), (777, 67, {}), (600, 80, {"tau_f": 0.8}), (130, 20, {})]


def test_threads_step_their_own_lattices():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_05264_gb300 import lbm as L

    def lattice(nx, ny, extra):
        p = PP.resolve(PP.default_params(geometry="channel", u_in=0.02, dTheat_R=0.05, heat_on_step=5, heater_x0=nx // 3,
                                         heater_len=20, g_a=1e-5, **extra), nx)
        lat = L.Lattice(nx, ny, "fp32")
        lat.set_params(p)
        lat.init_fields(*I.smooth_random(nx, ny, 5.95, 0.9 * PP.Tc(p), seed=nx, drho=0.002, du=0.004, dT=0.002))
        assert lat.step_loop == "persistent"
        return lat

    alone = [lattice(*s) for s in SIZES]
    for lat in alone:
        lat.step(CALLS)
    lats, failed = [lattice(*s) for s in SIZES], []
    ready = threading.Barrier(len(lats))

    def work(lat):
        ready.wait()
        try:
            for _ in range(CALLS):
                lat.step_async(1)
            lat.sync()
        except L.LbmError as e:
            failed.append(str(e))

    threads = [threading.Thread(target=work, args=(lat,)) for lat in lats]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    for a, b in zip(lats, alone):
        for x, y in zip(a.populations(), b.populations()):
            assert np.array_equal(x, y)
