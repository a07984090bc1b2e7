"""The FP64 step's reciprocal rounds as well as two Newton-Raphson steps do.

One step of Householder's method, 1/x = y (1 + e + e^2 + e^3) from y = rcp.approx(x) with |e| < 2^-19,
leaves e^4 < 2^-76 and about 2^-71 from the rounding of its polynomial before the last rounding: at most
0.5 + 2^-17 ulp.  Checked with room for an 80-bit reference (0.501; cut after e^2 it is 0.506), over the
ranges of the step.
"""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from test_gpu_fastmath import inputs, probe_lib, ulp_error  # noqa: F401


def test_fp64_reciprocal_is_rounded_once(probe_lib):  # noqa: F811
    if np.finfo(np.longdouble).eps >= np.finfo(np.float64).eps:
        pytest.skip("the host has no wider floating-point format than double for the reference")
    x = inputs()
    tx = torch.from_numpy(x).to("cuda")
    outs = [torch.empty_like(tx) for _ in range(3)]
    assert probe_lib.run_probe(*[ctypes.c_void_p(t.data_ptr()) for t in [tx] + outs], x.size) == 0
    assert ulp_error(outs[0].cpu().numpy(), 1.0 / x.astype(np.longdouble)).max() <= 0.501
