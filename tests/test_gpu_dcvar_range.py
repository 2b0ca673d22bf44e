"""The outer residual with a variable 2D stencil where magnitudes leave the exponent
range that the integer form takes (biased exponents 128 to 1900): those chunks are
done in FP64.

1025^2, the smallest size alone on the integer form. Tolerances as in the tests of
that form: the scaled problem's residual is the scaled residual, to the rounding
of two FP64 evaluations (1e-13); the defect, where FP32 can hold it, to FP32's.
"""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu
N = 1025


def outer(k, f, u):
    need_gpu()
    from paper_1406_5369_gb300 import Solver
    s = Solver(2, N, k=k, precision="fp32_dc")
    s.set_rhs(f)
    s.set_solution(u)
    return s.residual_norm(), s.get_field(0, "f")


def fields():
    k = np.exp(3.0 * synth.uniform(51, (N, N)))
    f, u = synth.uniform_rhs(2, N, 55), synth.uniform(56, (N, N))
    u[0], u[-1], u[:, 0], u[:, -1] = 0, 0, 0, 0
    return k, f, u


# u at 2^-930 (biased 93) and 2^890 (1913); k keeps the squares in FP64's range
# (and its own: the faces' harmonic means multiply two coefficients)
@pytest.mark.parametrize("shift,back", [(-930, 500), (890, -480)])
def test_solution_outside_the_range(shift, back):
    k, f, u = fields()
    n0, _ = outer(k, f, u)
    n1, _ = outer(np.ldexp(k, back), np.ldexp(f, shift + back), np.ldexp(u, shift))
    assert abs(np.ldexp(n1, -shift - back) - n0) <= 1e-13 * n0


def test_small_rows_before_ordinary_ones():
    """Chunks that begin below the range and go on inside it."""
    k, f, u = fields()
    u *= np.ldexp(1.0, np.where(np.arange(N) % 37 < 20, -940, 0))[:, None]
    norm, d = outer(k, f, u)
    r = oracle.residual(u, f, faces=oracle.node_faces(k))
    assert abs(norm - oracle.norm(r)) <= 1e-12 * norm
    assert np.abs(d - r)[1:-1, 1:-1].max() <= 2.0 ** -22 * np.abs(r).max()
