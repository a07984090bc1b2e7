"""The columns beyond a channel's outlet do not decide its stability.

A strip's lanes outside the lattice read the end column in place of their own.  With opposing vertical
velocities (0.45) two rows apart in the last column such a node would collect a density outside the
equation of state (9.8 against 1/b = 10.5, psi radicand negative), while every node of the lattice stays
between 5.7 and 6.3: the oracle steps it, and so does the library, with one launch per step and with
the flat launch.
"""
import numpy as np
import pytest

import oracle
from paper_2009_05264_gb300 import params as PP

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx", [130, 131])
@pytest.mark.parametrize("loop", ["launches", "auto"])
def test_nodes_outside_the_lattice_are_not_checked(nx, loop):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2009_05264_gb300 import lbm as L

    ny = 20
    p = PP.resolve(PP.default_params(geometry="channel", u_in=0.02, dTheat_R=0.05, heat_on_step=5, heater_x0=40,
                                     heater_len=10, g_a=0.0), nx)
    fields = [np.full((ny, nx), v) for v in (5.95, 0.02, 0.0, 0.9 * oracle.Tc(p))]
    fields[2][9, -1], fields[2][11, -1] = 0.45, -0.45
    orc = oracle.Oracle(nx, ny, p)
    orc.init_fields(*fields)
    assert orc.step(2) == 0
    lat = L.Lattice(nx, ny, "fp32")
    lat.set_params(p)
    lat.set_step_loop(loop)
    lat.init_fields(*fields)
    lat.step(2)  # the second step pulls from the first one's populations
    rho, ref = lat.fields()["rho"], orc.fields()["rho"]
    assert np.abs(rho - ref).max() < 1e-5 * np.abs(ref).max()
