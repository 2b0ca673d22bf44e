"""Smoothers of the FP32 and BF16 levels divide by the diagonal, rounding once: from
u = 0 and with omega = 1 a sweep's first values are f / diag as FP32 rounds it. (A
product with the rounded reciprocal differs in the last place at a quarter of the
nodes.)"""
import numpy as np
import pytest

import synth
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("smoother", ["rbgs", "jacobi"])
@pytest.mark.parametrize("n", [33, 129])
def test_first_sweep_from_zero(n, smoother):
    need_gpu()
    from paper_1406_5369_gb300 import Solver
    c = (0.7, 1.4)
    s = Solver(2, n, stencil=c + (1.0,), smoother=smoother, omega=1.0, precision="fp32_dc")
    f = synth.uniform_rhs(2, n, 97).astype(np.float32)
    s.set_field(0, "f", f.astype(np.float64))
    s.set_field(0, "u", np.zeros((n, n)))
    s.smooth(0, 1)
    h = 1.0 / (n - 1)
    want = f / np.float32(2.0 * (c[0] + c[1]) * (1.0 / (h * h)))
    got = s.get_field(0, "u")[1:-1, 1:-1].astype(np.float32)
    i = np.arange(1, n - 1)
    mine = np.ones((n - 2, n - 2), bool) if smoother == "jacobi" else (i[:, None] + i[None]) % 2 == 0
    assert np.array_equal(got[mine], want[1:-1, 1:-1][mine])
