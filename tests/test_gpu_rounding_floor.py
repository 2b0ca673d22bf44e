"""Solves carried on to the FP64 rounding floor come to rest where the oracle's
FP64 cycles do: tolerances that an FP64 solve can reach stay reachable.

At the floor the residual is A times the rounding of the stored solution, half a
unit in the last place of each value, and a sweep that rounds each new value
once leaves just that. The factor 1.4 allows the rounding of the sweeps before
it to add as much again in the sum of squares; a last sweep that rounds sums of
neighbours has 1.5 (few cells) to 3.8 times the oracle's. Both floors are means
over the last cycles.
"""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu

SM = {"rbgs": oracle.RBGS, "jacobi": oracle.JACOBI}


def compare(hist, rho):
    got, want = np.mean(hist[-8:]), np.mean(rho[-8:])
    assert got <= 1.4 * want, (got, want)


# 8: every level in one block; 16 and up: a kernel per sweep on the finest level
@pytest.mark.parametrize("n,bc,sigma,smoother,omega,nu,c", [
    (8, "neumann", 1.0, "rbgs", 1.0, (2, 2), (1.0, 1.0, 1.0)),
    (8, "dirichlet", 1.0, "jacobi", 0.8, (2, 1), (1.0, 1.0, 0.7)),
    (16, "neumann", 1.0, "rbgs", 1.0, (2, 2), (1.0, 1.0, 1.0)),
    (32, "dirichlet", 1.0, "jacobi", 0.8, (2, 2), (1.0, 0.8, 1.2)),
    (64, "neumann", 1.0, "rbgs", 1.1, (2, 2), (1.0, 1.0, 1.0)),
    (64, "dirichlet", 1.0, "rbgs", 1.0, (2, 1), (1.0, 1.0, 1.0)),
])
def test_cell_3d(n, bc, sigma, smoother, omega, nu, c):
    need_gpu()
    from paper_1406_5369_gb300 import CCSolver
    f = synth.uniform(71, (n, n, n))
    kw = dict(c=c, sigma=sigma, bc=bc, omega=omega, nu1=nu[0], nu2=nu[1])
    s = CCSolver(3, n, smoother=smoother, maxit=40, **kw)
    s.set_rhs(f)
    s.set_solution(None)
    _, _, hist = s.solve(0.0, raise_on_noconv=False)
    ref = oracle.CCHierarchy(3, n, smoother=SM[smoother], **kw)
    ref.set_rhs(f)
    ref.set_u(np.zeros_like(f))
    compare(hist, ref.solve(0.0, 40))


# the cluster cycle: one block (up to 17, 16 cells), bands over the blocks above
@pytest.mark.parametrize("n,smoother,omega,nu,c", [
    (17, "rbgs", 1.0, (2, 1), (0.8, 1.3)),
    (33, "rbgs", 1.1, (2, 2), (0.8, 1.3)),
    (33, "jacobi", 0.8, (2, 1), (1.0, 1.0)),
    (65, "jacobi", 0.8, (2, 2), (1.0, 1.0)),
    (65, "rbgs", 1.0, (2, 2), (0.8, 1.3)),
    (129, "rbgs", 1.0, (2, 1), (0.8, 1.3)),
    (129, "jacobi", 0.8, (1, 3), (1.0, 1.0)),
])
def test_node_2d_cluster(n, smoother, omega, nu, c):
    need_gpu()
    from paper_1406_5369_gb300 import Solver
    f = synth.uniform_rhs(2, n, 72)
    s = Solver(2, n, smoother=smoother, omega=omega, nu1=nu[0], nu2=nu[1], stencil=c + (1.0,), maxit=40)
    s.set_rhs(f)
    _, _, hist = s.solve(0.0, raise_on_noconv=False)
    ref = oracle.Hierarchy(2, n, c=c, smoother=SM[smoother], omega=omega, nu1=nu[0], nu2=nu[1])
    ref.set_rhs(f)
    ref.set_u(np.zeros_like(f))
    compare(hist, ref.solve(0.0, 40))


@pytest.mark.parametrize("n,bc,sigma,smoother,omega,nu,c", [
    (16, "neumann", 1.0, "rbgs", 1.0, (2, 2), (1.0, 1.0)),
    (32, "neumann", 1.0, "rbgs", 1.0, (2, 2), (1.0, 1.0)),
    (64, "dirichlet", 1.0, "rbgs", 1.1, (2, 1), (1.0, 1.0)),
    (64, "neumann", 500.0, "rbgs", 1.0, (2, 2), (0.9, 1.2)),
    (128, "neumann", 1.0, "jacobi", 0.8, (2, 2), (1.0, 1.0)),
    (128, "dirichlet", 1.0, "rbgs", 1.0, (2, 2), (1.0, 1.0)),
])
def test_cell_2d_cluster(n, bc, sigma, smoother, omega, nu, c):
    need_gpu()
    from paper_1406_5369_gb300 import CCSolver
    f = synth.uniform(73, (n, n))
    kw = dict(c=c, sigma=sigma, bc=bc, omega=omega, nu1=nu[0], nu2=nu[1])
    s = CCSolver(2, n, smoother=smoother, maxit=40, **kw)
    s.set_rhs(f)
    s.set_solution(None)
    _, _, hist = s.solve(0.0, raise_on_noconv=False)
    ref = oracle.CCHierarchy(2, n, smoother=SM[smoother], **kw)
    ref.set_rhs(f)
    ref.set_u(np.zeros_like(f))
    compare(hist, ref.solve(0.0, 40))


@pytest.mark.parametrize("n,tau,smoother,omega,nu", [
    (64, 1e-3, "jacobi", 0.8, (2, 2)),
    (128, 1e-3, "rbgs", 1.1, (2, 1)),
    (256, 1e-3, "jacobi", 0.8, (3, 2)),
])
def test_complex_diffusion(n, tau, smoother, omega, nu):
    need_gpu()
    from paper_1406_5369_gb300 import CDSolver
    un = synth.uniform(74, (n, n)) + 0.02j * synth.uniform(75, (n, n))
    s = CDSolver(n, tau=tau, theta=np.pi / 30, kappa=0.1, smoother=smoother, omega=omega, nu1=nu[0], nu2=nu[1], maxit=40)
    _, _, hist = s.time_step(un, 0.0, raise_on_noconv=False)
    ref = oracle.CDHierarchy(n, tau, np.pi / 30, 0.1, smoother=SM[smoother], omega=omega, nu1=nu[0], nu2=nu[1])
    _, rho = ref.time_step(un, 0.0, 40)
    compare(hist, rho)
