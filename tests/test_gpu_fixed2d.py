"""The fixed-point 2D passes and the other FP64 cycles against the oracle's FP64
V-cycles and the per-operator kernels (fuse=False).

Tolerances: per-cycle relative residuals to 1e-12 (the bound of the FP64
path); solutions to 1e-12 of their largest value (two FP64 evaluations of the
same cycles, each with a rounding error of a few 1e-16 per sweep).
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
    return Solver(2, n, **kw)


# 65: two strips; 129, 257, 513: ragged last strips and row chunks; 1025: several chunks per strip
@pytest.mark.parametrize("n,smoother,omega,nu,c,rows", [
    (65, "rbgs", 1.0, (2, 2), (1.0, 1.0), 0),
    (129, "jacobi", 0.8, (1, 2), (1.0, 1.0), 0),
    (257, "rbgs", 1.15, (3, 2), (1.0, 1.0), 8),
    (257, "jacobi", 0.75, (3, 3), (0.7, 1.4), 16),
    (513, "rbgs", 1.0, (1, 3), (1.3, 0.8), 0),
    (513, "rbgs", 0.9, (2, 1), (3.0, 3.0), 24),
    (1025, "jacobi", 0.8, (2, 2), (1.0, 1.0), 0),
    (1025, "rbgs", 1.0, (4, 5), (1.0, 1.0), 0),
    (513, "rbgs", 1.9, (2, 2), (1.0, 1.0), 0),     # growth bound: stays on the FP64 kernels
    (257, "rbgs", 1.0, (2, 2), (1.0, 1e-4), 0),    # so do very different coefficients
])
def test_cycles_match_oracle(n, smoother, omega, nu, c, rows):
    f = synth.uniform_rhs(2, n, 11)
    b = synth.uniform(3, (n, n)) * 1e-3
    s = solver(n, smoother=smoother, omega=omega, nu1=nu[0], nu2=nu[1], stencil=c + (1.0,), maxit=3,
               dirichlet=b, tile_rows=rows, cluster_max_n=33)
    s.set_rhs(f)
    _, _, hist = s.solve(0.0, raise_on_noconv=False)
    ref = oracle.Hierarchy(2, n, c=c, smoother=SM[smoother], omega=omega, nu1=nu[0], nu2=nu[1])
    u0 = np.array(b)
    u0[1:-1, 1:-1] = 0.0
    ref.set_u(u0)
    ref.set_rhs(f)
    rho = ref.solve(0.0, 3)
    assert np.max(np.abs(hist - rho) / np.maximum(1.0, rho)) <= 1e-12, (hist, rho)
    u = s.get_solution()
    assert rel_err(u, ref.get_u()) <= 1e-12
    assert np.array_equal(u[0], b[0]) and np.array_equal(u[:, -1], b[:, -1])  # boundary values stay


@pytest.mark.parametrize("smoother,omega", [("rbgs", 1.0), ("jacobi", 0.8)])
@pytest.mark.parametrize("shift", [-980, -600, 600, 900])
def test_scaling_by_powers_of_two(smoother, omega, shift):
    """The scale follows the data; magnitudes outside the exponent range are done in FP64."""
    n = 257
    f = synth.uniform_rhs(2, n, 5)
    got = []
    for e in (0, shift):
        s = solver(n, smoother=smoother, omega=omega, nu1=2, nu2=2)
        s.set_rhs(np.ldexp(f, e))
        s.vcycle()
        got.append(np.ldexp(s.get_solution(), -e))
    assert rel_err(got[1], got[0]) <= 1e-13


def test_wide_range_of_magnitudes():
    """Rows of very different size in one strip, growing and falling: the window is rescaled."""
    n = 513
    f = synth.uniform_rhs(2, n, 6) * np.ldexp(1.0, (np.arange(n) * 7) % 90 - 45)[:, None]
    out = []
    for fuse in (True, False):
        s = solver(n, nu1=2, nu2=2, fuse=fuse, cluster_max_n=33)
        s.set_rhs(f)
        s.vcycle()
        s.vcycle()
        out.append(s.get_solution())
    assert rel_err(out[0], out[1]) <= 1e-13


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_values(bad):
    n = 513
    f = synth.uniform_rhs(2, n, 8)
    edge = np.array(f)
    edge[0], edge[-1], edge[:, 0], edge[:, -1] = bad, bad, bad, bad
    hole = np.array(f)
    hole[200, 300] = bad
    res = {}
    for name, rhs in (("plain", f), ("edge", edge), ("hole", hole)):
        for fuse in (True, False):
            s = solver(n, nu1=2, nu2=2, fuse=fuse, cluster_max_n=33)
            s.set_rhs(rhs)
            s.vcycle()
            res[name, fuse] = s.get_solution()
    # the right-hand side of boundary nodes is not read
    assert np.array_equal(res["edge", True], res["plain", True])
    assert np.array_equal(np.isfinite(res["hole", True]), np.isfinite(res["hole", False]))
    assert not np.isfinite(res["hole", True]).all()


# 64: one strip and a ragged one; 512, 1024: several chunks; sigma h^2 from 1e-6 to 0.8 and zero
@pytest.mark.parametrize("n,bc,sigma,smoother,omega,nu,c", [
    (64, "neumann", 3000.0, "rbgs", 1.0, (2, 2), (1.0, 1.0)),
    (128, "dirichlet", 0.0, "rbgs", 1.1, (2, 1), (1.0, 1.0)),
    (256, "neumann", 1.0, "jacobi", 0.8, (3, 2), (1.0, 1.0)),
    (512, "dirichlet", 50.0, "rbgs", 1.0, (1, 3), (0.8, 1.25)),
    (512, "neumann", 10.0, "jacobi", 0.8, (2, 2), (1.25, 0.9)),
    (1024, "neumann", 1.0, "rbgs", 1.0, (2, 2), (1.0, 1.0)),
    (64, "neumann", 1e5, "rbgs", 1.0, (2, 2), (1.0, 1.0)),  # sigma h^2 = 24: stays on the FP64 kernels
])
def test_cell_cycles_match_oracle(n, bc, sigma, smoother, omega, nu, c):
    need_gpu()
    from paper_1406_5369_gb300 import CCSolver
    f, u0 = synth.uniform(21, (n, n)) - 0.5, synth.uniform(22, (n, n))
    s = CCSolver(2, n, c=c, sigma=sigma, bc=bc, smoother=smoother, omega=omega, nu1=nu[0], nu2=nu[1], maxit=3)
    s.set_rhs(f)
    s.set_solution(u0)
    _, _, hist = s.solve(0.0, raise_on_noconv=False)
    ref = oracle.CCHierarchy(2, n, c=c, sigma=sigma, bc=bc, smoother=SM[smoother], omega=omega, nu1=nu[0], nu2=nu[1])
    ref.set_rhs(f)
    ref.set_u(u0)
    rho = ref.solve(0.0, 3)
    assert np.max(np.abs(hist - rho) / np.maximum(1.0, rho)) <= 1e-12, (hist, rho)
    assert rel_err(s.get_field(0, "u"), ref.get_u()) <= 1e-12


# every depth of the cluster cycle, up to its largest level (257), alone and below the streaming passes
@pytest.mark.parametrize("n,smoother,omega,nu,c,nc,top", [
    (5, "rbgs", 1.0, (2, 1), (1.0, 1.0), 3, 0),
    (9, "jacobi", 0.8, (1, 2), (1.0, 2.0), 5, 0),
    (17, "rbgs", 1.2, (0, 2), (1.0, 1.0), 9, 0),
    (33, "jacobi", 0.7, (2, 1), (1.0, 1.0), 3, 0),
    (65, "rbgs", 1.0, (2, 0), (1.5, 0.5), 3, 0),
    (65, "jacobi", 0.8, (3, 2), (1.0, 1.0), 9, 0),
    (129, "rbgs", 1.0, (2, 1), (1.0, 1.0), 3, 0),
    (129, "jacobi", 0.8, (1, 1), (1.0, 1.0), 5, 0),
    (257, "rbgs", 1.1, (2, 2), (1.0, 1.0), 9, 257),
    (513, "jacobi", 0.8, (1, 2), (1.0, 1.0), 3, 0),
])
def test_cluster_cycle_matches_oracle(n, smoother, omega, nu, c, nc, top):
    f = synth.uniform_rhs(2, n, 31)
    b = synth.uniform(32, (n, n)) * 0.1
    s = solver(n, smoother=smoother, omega=omega, nu1=nu[0], nu2=nu[1], stencil=c + (1.0,), maxit=3, dirichlet=b,
               coarsest_n=nc, cluster_max_n=top)
    s.set_rhs(f)
    _, _, hist = s.solve(0.0, raise_on_noconv=False)
    ref = oracle.Hierarchy(2, n, c=c, smoother=SM[smoother], omega=omega, nu1=nu[0], nu2=nu[1], coarsest_n=nc)
    u0 = np.array(b)
    u0[1:-1, 1:-1] = 0.0
    ref.set_u(u0)
    ref.set_rhs(f)
    rho = ref.solve(0.0, 3)
    assert np.max(np.abs(hist - rho) / np.maximum(1.0, rho)) <= 1e-12, (hist, rho)
    u = s.get_solution()
    assert rel_err(u, ref.get_u()) <= 1e-12
    assert np.array_equal(u[0], b[0]) and np.array_equal(u[:, -1], b[:, -1])


@pytest.mark.parametrize("n,bc,sigma,smoother,omega,nu,nc", [
    (2, "dirichlet", 0.0, "rbgs", 1.0, (2, 1), 1),
    (4, "neumann", 5.0, "jacobi", 0.8, (1, 2), 1),
    (8, "dirichlet", 1.0, "rbgs", 1.2, (0, 2), 4),
    (32, "neumann", 100.0, "rbgs", 1.0, (2, 2), 2),
    (64, "neumann", 1.0, "jacobi", 0.8, (3, 2), 1),
    (64, "dirichlet", 2000.0, "rbgs", 1.0, (1, 0), 4),
    (128, "dirichlet", 0.0, "jacobi", 0.8, (1, 2), 2),
    (128, "neumann", 0.01, "rbgs", 1.0, (2, 2), 1),
])
def test_cell_cluster_cycle_matches_oracle(n, bc, sigma, smoother, omega, nu, nc):
    need_gpu()
    from paper_1406_5369_gb300 import CCSolver
    c = (1.0, 0.7)
    f, u0 = synth.uniform(21, (n, n)) - 0.5, synth.uniform(22, (n, n))
    s = CCSolver(2, n, c=c, sigma=sigma, bc=bc, smoother=smoother, omega=omega, nu1=nu[0], nu2=nu[1], maxit=3,
                 coarsest_n=nc)
    s.set_rhs(f)
    s.set_solution(u0)
    _, _, hist = s.solve(0.0, raise_on_noconv=False)
    ref = oracle.CCHierarchy(2, n, c=c, sigma=sigma, bc=bc, smoother=SM[smoother], omega=omega, nu1=nu[0],
                             nu2=nu[1], coarsest_n=nc)
    ref.set_rhs(f)
    ref.set_u(u0)
    rho = ref.solve(0.0, 3)
    assert np.max(np.abs(hist - rho) / np.maximum(1.0, rho)) <= 1e-12, (hist, rho)
    assert rel_err(s.get_field(0, "u"), ref.get_u()) <= 1e-12


# 3D cells: sums over the outer faces of coarse cells, first half-sweep from zero
@pytest.mark.parametrize("n,bc,sigma,smoother,omega,nu,c", [
    (64, "neumann", 3000.0, "rbgs", 1.0, (2, 2), (1.0, 1.0, 1.0)),
    (64, "dirichlet", 0.0, "rbgs", 1.1, (2, 1), (1.0, 1.0, 1.0)),
    (128, "neumann", 1.0, "jacobi", 0.8, (3, 2), (1.0, 1.0, 1.0)),
    (128, "dirichlet", 100.0, "rbgs", 1.0, (1, 3), (0.8, 1.25, 1.0)),
    (64, "neumann", 10.0, "jacobi", 0.8, (2, 2), (1.25, 0.9, 0.9)),
    (8, "neumann", 1.0, "rbgs", 1.0, (0, 2), (1.0, 1.0, 1.0)),
    (8, "dirichlet", 3.0, "jacobi", 0.8, (2, 0), (1.0, 2.0, 1.0)),
    (16, "neumann", 2.0, "jacobi", 0.8, (3, 2), (1.0, 1.0, 1.0)),
    (32, "dirichlet", 0.0, "rbgs", 1.3, (1, 2), (1.0, 1.0, 0.6)),
    (4, "dirichlet", 0.0, "jacobi", 0.8, (1, 0), (1.0, 1.0, 1.0)),
])
def test_cell_3d_cycles_match_oracle(n, bc, sigma, smoother, omega, nu, c):
    need_gpu()
    from paper_1406_5369_gb300 import CCSolver
    f, u0 = synth.uniform(21, (n, n, n)) - 0.5, synth.uniform(22, (n, n, n))
    s = CCSolver(3, n, c=c, sigma=sigma, bc=bc, smoother=smoother, omega=omega, nu1=nu[0], nu2=nu[1], maxit=2)
    s.set_rhs(f)
    s.set_solution(u0)
    _, _, hist = s.solve(0.0, raise_on_noconv=False)
    ref = oracle.CCHierarchy(3, n, c=c, sigma=sigma, bc=bc, smoother=SM[smoother], omega=omega, nu1=nu[0], nu2=nu[1])
    ref.set_rhs(f)
    ref.set_u(u0)
    rho = ref.solve(0.0, 2)
    assert np.max(np.abs(hist - rho) / np.maximum(1.0, rho)) <= 1e-12, (hist, rho)
    assert rel_err(s.get_field(0, "u"), ref.get_u()) <= 1e-12
