"""Screened cell problems, whose solutions decay by orders of magnitude over a few
cells, keep their relative precision where FP64 sweeps reach it.

The data depend on one coordinate only, so the solution is that of a tridiagonal
system, solved here in extended precision. Carried on to the rounding floor, FP64
V-cycles come within n^2 2^-53 / 100 = 3e-13 of the solution (n = 512), relative
to the value itself, down to 1e-11 of the largest one; the bound is 1e-12.
"""
import numpy as np
import pytest

from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def tridiagonal(d, k, f):
    """-k u[i-1] + d[i] u[i] - k u[i+1] = f[i], without cancellation for f >= 0."""
    n = len(f)
    d, k = np.asarray(d, np.longdouble), np.longdouble(k)
    c, g = np.zeros(n, np.longdouble), np.zeros(n, np.longdouble)
    for i in range(n):
        m = d[i] - (k * c[i - 1] if i else 0)
        c[i], g[i] = k / m, (f[i] + (k * g[i - 1] if i else 0)) / m
    for i in range(n - 2, -1, -1):
        g[i] += c[i] * g[i + 1]
    return g


@pytest.mark.parametrize("n,reaction", [(256, 0.9), (512, 0.05), (512, 0.3), (512, 0.005), (1024, 0.02)])
@pytest.mark.parametrize("axis", [0, 1])
def test_relative_precision(n, reaction, axis):
    need_gpu()
    from paper_1406_5369_gb300 import CCSolver
    k = float(n * n)
    f1 = np.zeros(n)
    f1[:4] = k
    d = np.full(n, (2 + reaction) * k)
    d[0] = d[-1] = (1 + reaction) * k
    want = tridiagonal(d, k, f1)
    f = np.repeat(f1[:, None], n, 1) if axis == 0 else np.repeat(f1[None], n, 0)
    s = CCSolver(2, n, sigma=reaction * k, nu1=2, nu2=2, maxit=40)
    s.set_rhs(f)
    s.set_solution(None)
    s.solve(0.0, raise_on_noconv=False)
    u = s.get_solution()
    seen = want >= 1e-11 * want.max()
    w = want[:, None] if axis == 0 else want[None]
    m = seen[:, None] if axis == 0 else seen[None]
    err = np.where(m, np.abs(u - w) / w, 0)
    assert err.max() <= 1e-12, float(err.max())
