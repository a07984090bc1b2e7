"""Parameters that are refused leave the lattice as it was.

A wall density whose psi is undefined (Eq. 11) passes the range checks and is refused while the
descriptor is formed: the call reports LBM_EINVAL, and the lattice goes on stepping with the parameters
and the state that it had, bit for bit, in every kernel form that takes its descriptor as a launch
parameter.  The same for a checkpoint whose parameters are refused.
"""
import numpy as np
import pytest

from paper_2009_05264_gb300 import inputs as I
from paper_2009_05264_gb300 import params as PP

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,loop,extra", [
    ("fp32", "auto", {}), ("fp32", "auto", {"bubble_stats": 1}), ("fp32", "launches", {}),
    ("fp32", "launches", {"source_model": 1}), ("fp64", "auto", {}), ("fp64", "launches", {"bubble_stats": 1})])
def test_refused_parameters_change_nothing(prec, loop, extra):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_05264_gb300 import lbm as L

    nx, ny = 130, 20
    p = PP.resolve(PP.default_params(geometry="channel", u_in=0.02, dTheat_R=0.05, heat_on_step=5, heater_x0=40,
                                     heater_len=10, g_a=1e-5, **extra), nx)
    fields = I.smooth_random(nx, ny, 5.95, 0.9 * PP.Tc(p), seed=3, drho=0.002, du=0.004, dT=0.002)
    lat, ref = L.Lattice(nx, ny, prec), L.Lattice(nx, ny, prec)
    for a in (lat, ref):
        a.set_params(p)
        a.set_step_loop(loop)
        a.init_fields(*fields)
        a.step(4)
    with pytest.raises(L.LbmError) as err:
        lat.set_params(dict(p, rho_w=9.5))
    assert err.value.status == 1 and "psi" in str(err.value)  # LBM_EINVAL
    blob = bytearray(ref.save_state())
    at = L.LbmParams.rho_w.offset + 24  # behind the header's magic, sizes, precision and version
    assert np.frombuffer(blob, np.float64, 1, at)[0] == p["rho_w"]
    np.frombuffer(blob, np.float64, 1, at)[:] = 9.5
    with pytest.raises(L.LbmError):
        lat.load_state(bytes(blob))
    for a in (lat, ref):
        a.step(7)
    assert lat.step_count == 11
    for x, y in zip(lat.populations(), ref.populations()):
        assert np.array_equal(x, y)
