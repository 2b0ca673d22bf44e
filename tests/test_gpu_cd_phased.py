"""A step's V-cycles on real face weights with one phase against the same
cycles on complex faces (reading a face switches a context to those).

Tolerance 1e-13 of the largest value: both are FP64 evaluations of the same
cycles, each with a few 1e-16 of rounding per sweep.
"""
import numpy as np
import pytest

import synth
from gpu_util import need_gpu, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 4, 16, 64, 512])
@pytest.mark.parametrize("smoother,omega,nu", [
    ("rbgs", 1.0, (2, 2)), ("rbgs", 1.3, (0, 2)), ("jacobi", 0.8, (2, 1)), ("jacobi", 0.7, (1, 0)), ("jacobi", 1.0, (3, 3))])
def test_phased_cycles_match_complex_ones(n, smoother, omega, nu):
    need_gpu()
    from paper_1406_5369_gb300 import CDSolver
    un = synth.uniform(41, (n, n)) + 1j * (synth.uniform(42, (n, n)) - 0.5) * 0.2
    out = []
    for phased in (True, False):
        s = CDSolver(n, tau=1e-3, smoother=smoother, omega=omega, nu1=nu[0], nu2=nu[1])
        s.begin_step(un)
        if not phased:
            s.get_field(0, "gx")
        s.vcycle()
        r1 = s.residual_norm()
        s.vcycle()
        out.append((s.get_field(0, "u"), r1, s.residual_norm()))
    scale = np.linalg.norm(un)
    assert rel_err(out[0][0], out[1][0]) <= 1e-13
    assert abs(out[0][1] - out[1][1]) <= 1e-12 * scale and abs(out[0][2] - out[1][2]) <= 1e-12 * scale


def test_right_hand_side_set_by_the_caller():
    """Setting f after begin_step takes effect on either kind of faces."""
    need_gpu()
    from paper_1406_5369_gb300 import CDSolver
    n = 64
    un = synth.uniform(43, (n, n)) + 0.1j * synth.uniform(44, (n, n))
    f = synth.uniform(45, (n, n)) + 0j
    out = []
    for phased in (True, False):
        s = CDSolver(n, tau=1e-3)
        s.begin_step(un)
        if not phased:
            s.get_field(0, "gy")
        s.set_field(0, "f", f)
        s.vcycle()
        out.append(s.get_field(0, "u"))
    assert rel_err(out[0], out[1]) <= 1e-13
