"""The fixed-point 3D passes of the FP64 levels against the oracle's FP64
V-cycles and the per-operator kernels (fuse=False). Tolerances as for the 2D
passes: residual histories to 1e-12, solutions to 1e-12 of their largest value.
"""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import need_gpu, rel_err

pytestmark = pytest.mark.gpu

SM = {"rbgs": oracle.RBGS, "jacobi": oracle.JACOBI}


def solver(n, **kw):
    need_gpu()
    from paper_1406_5369_gb300 import Solver
    return Solver(3, n, **kw)


# 257: the smallest level that takes the passes (ragged tiles and plane chunks); 65 and 129 keep FP64 kernels
@pytest.mark.parametrize("n,smoother,omega,nu,c", [
    (65, "jacobi", 6.0 / 7.0, (1, 3), (1.0, 1.0, 1.0)),
    (129, "rbgs", 1.0, (3, 2), (0.7, 1.0, 1.4)),
    (257, "rbgs", 1.0, (2, 2), (1.0, 1.0, 1.0)),
    (257, "rbgs", 1.15, (1, 1), (0.7, 1.0, 1.4)),
    (257, "jacobi", 0.8, (2, 1), (1.3, 1.3, 0.9)),
    (257, "jacobi", 6.0 / 7.0, (1, 3), (3.0, 3.0, 3.0)),
    (257, "rbgs", 1.0, (2, 1), (1.0, 1.0, 1e-4)),    # very different coefficients: stays on the FP64 kernels
])
def test_cycles_match_oracle(n, smoother, omega, nu, c):
    f = synth.uniform_rhs(3, n, 11)
    b = synth.uniform(3, (n, n, n)) * 1e-3
    s = solver(n, smoother=smoother, omega=omega, nu1=nu[0], nu2=nu[1], stencil=c, maxit=1, dirichlet=b)
    s.set_rhs(f)
    _, _, hist = s.solve(0.0, raise_on_noconv=False)
    ref = oracle.Hierarchy(3, n, c=c, smoother=SM[smoother], omega=omega, nu1=nu[0], nu2=nu[1],
                           mt=True)
    u0 = np.array(b)
    u0[1:-1, 1:-1, 1:-1] = 0.0
    ref.set_u(u0)
    ref.set_rhs(f)
    rho = ref.solve(0.0, 1)
    assert np.max(np.abs(hist - rho) / np.maximum(1.0, rho)) <= 1e-12, (hist, rho)
    u = s.get_solution()
    assert rel_err(u, ref.get_u()) <= 1e-12
    for ax in range(3):
        assert np.array_equal(np.take(u, (0, n - 1), ax), np.take(b, (0, n - 1), ax))  # boundary values stay


@pytest.mark.parametrize("smoother,omega", [("rbgs", 1.0), ("jacobi", 0.8)])
@pytest.mark.parametrize("shift", [-980, 900])
def test_scaling_by_powers_of_two(smoother, omega, shift):
    n = 257
    f = synth.uniform_rhs(3, n, 5)
    got = []
    for e in (0, shift):
        s = solver(n, smoother=smoother, omega=omega, nu1=2, nu2=2)
        s.set_rhs(np.ldexp(f, e))
        s.vcycle()
        got.append(np.ldexp(s.get_solution(), -e))
    assert rel_err(got[1], got[0]) <= 1e-13


@pytest.mark.parametrize("smoother,omega", [("rbgs", 1.0), ("jacobi", 0.8)])
def test_wide_range_of_magnitudes(smoother, omega):
    """Planes of very different size, growing and falling: the window is rescaled."""
    n = 257
    f = synth.uniform_rhs(3, n, 6) * np.ldexp(1.0, (np.arange(n) * 7) % 90 - 45)[:, None, None]
    out = []
    for fuse in (True, False):
        s = solver(n, nu1=2, nu2=2, smoother=smoother, omega=omega, fuse=fuse)
        s.set_rhs(f)
        s.vcycle()
        s.vcycle()
        out.append(s.get_solution())
    assert rel_err(out[0], out[1]) <= 1e-13


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_values(bad):
    n = 257
    f = synth.uniform_rhs(3, n, 8)
    edge = np.full((n, n, n), bad)
    edge[1:-1, 1:-1, 1:-1] = f[1:-1, 1:-1, 1:-1]
    hole = np.array(f)
    hole[20, 30, 40] = bad
    res = {}
    for name, rhs in (("plain", f), ("edge", edge), ("hole", hole)):
        for fuse in (True, False):
            s = solver(n, nu1=2, nu2=2, fuse=fuse)
            s.set_rhs(rhs)
            s.vcycle()
            res[name, fuse] = s.get_solution()
    # the right-hand side of boundary nodes is not read
    assert np.array_equal(res["edge", True], res["plain", True])
    assert np.array_equal(np.isfinite(res["hole", True]), np.isfinite(res["hole", False]))
    assert not np.isfinite(res["hole", True]).all()
