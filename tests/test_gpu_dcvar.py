"""The outer residual of defect correction with a variable 2D stencil against
the oracle's FP64 residual: the norm and the defect it leaves on level 0.

Tolerances: a flux is cut at 2^-58 of the largest |u| times the node's largest
coefficient (four fluxes, over h^2), so the residual is off by at most
2^-55 max|u| max(k) / h^2 and FP64 rounding of about as much; the defect is
FP32 (2^-23 relative, truncated or rounded).
"""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def outer(n, k, f, u, b=None, precision="fp32_dc"):
    need_gpu()
    from paper_1406_5369_gb300 import Solver
    s = Solver(2, n, k=k, dirichlet=b, precision=precision)
    s.set_rhs(f)
    s.set_solution(u)
    return s, s.residual_norm(), s.get_field(0, "f")


def coefficients(kind, n):
    g = synth.uniform(51, (n, n))
    if kind == "lognormal":
        return np.exp(2.0 * (g - 0.5) * 3.0)
    return np.where(g > 0.5, 1e8, 1.0)  # eight orders of magnitude between neighbours


# alone, 1025 is the smallest size on the integer kernel; the others keep the FP64 one
@pytest.mark.parametrize("n", [5, 9, 33, 129, 1025])
@pytest.mark.parametrize("kind", ["lognormal", "jump"])
@pytest.mark.parametrize("precision", ["fp32_dc", "bf16_dc"])
def test_outer_residual(n, kind, precision):
    k, f = coefficients(kind, n), synth.uniform_rhs(2, n, 52)
    b = synth.uniform(53, (n, n))
    u = np.array(b)
    u[1:-1, 1:-1] = synth.uniform(54, (n, n))[1:-1, 1:-1] * np.ldexp(1.0, np.arange(n) % 40 - 20)[1:-1, None]
    _, norm, d = outer(n, k, f, u, b, precision)
    r = oracle.residual(u, f, faces=oracle.node_faces(k))
    tol = 2.0 ** -52 * np.abs(u).max() * k.max() * (n - 1) ** 2
    ulp = 2.0 ** -22 if precision == "fp32_dc" else 2.0 ** -8
    err = np.abs(d - r)[1:-1, 1:-1]
    assert np.all(err <= tol + ulp * np.abs(r)[1:-1, 1:-1])
    assert abs(norm - oracle.norm(r)) <= tol * n + 1e-13 * norm


@pytest.mark.parametrize("shift", [-900, 700])
def test_magnitudes_outside_the_range(shift):
    """u beyond the exponent range of the scale: the same residual, scaled."""
    n = 1025
    k = coefficients("lognormal", n)
    f, u = synth.uniform_rhs(2, n, 55), synth.uniform(56, (n, n))
    u[0], u[-1], u[:, 0], u[:, -1] = 0, 0, 0, 0
    res = {}
    for e in (0, shift):
        s, norm, _ = outer(n, k, np.ldexp(f, e // 2), np.ldexp(u, e // 2))
        res[e] = np.ldexp(norm, -(e // 2))
    assert abs(res[0] - res[shift]) <= 1e-13 * res[0]


@pytest.mark.parametrize("where", ["u", "f"])
def test_non_finite_values_stay_where_they_are(where):
    n = 1025
    k = coefficients("lognormal", n)
    f, u = synth.uniform_rhs(2, n, 57), synth.uniform(58, (n, n))
    u[0], u[-1], u[:, 0], u[:, -1] = 0, 0, 0, 0
    {"u": u, "f": f}[where][70, 40] = np.inf
    _, _, d = outer(n, k, f, u)
    with np.errstate(invalid="ignore"):
        r = oracle.residual(u, f, faces=oracle.node_faces(k))
    assert np.array_equal(np.isfinite(d)[1:-1, 1:-1], np.isfinite(r)[1:-1, 1:-1])
    ok = np.isfinite(r)
    assert np.abs(d[ok] - r[ok]).max() <= 1e-6 * np.abs(r[ok]).max()


def test_batch_of_every_size():
    """Sizes on both kernels of the batch engine (257 is the smallest on the integer one)."""
    need_gpu()
    from paper_1406_5369_gb300 import BatchSolver, Solver
    sizes = [5, 9, 33, 65, 129, 257, 513, 1025]
    ks = [np.where(coefficients("jump", n) > 1, 30.0, 1.0) for n in sizes]
    fs = [synth.uniform_rhs(2, n, 70 + n) for n in sizes]
    solvers = [Solver(2, n, k=k, precision="fp32_dc", inner_cycles=2, maxit=40) for n, k in zip(sizes, ks)]
    b = BatchSolver(len(sizes))
    for s, f in zip(solvers, fs):
        s.set_rhs(f)
        s.set_solution(None)
        b.add(s)
    b.solve(1e-9, maxit=40)
    for s, f, k in zip(solvers, fs, ks):
        r = oracle.residual(s.get_solution(), f, faces=oracle.node_faces(k))
        assert oracle.norm(r) <= 1.01e-9 * oracle.norm(f)
