"""Batches of problems with variable coefficients of up to 257^2 form their outer
residuals in one launch, whatever their sizes (a second launch for the largest of
a few problems costs more than its kernel saves)."""
import numpy as np
import pytest

import synth
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def launches(sizes):
    from paper_1406_5369_gb300 import BatchSolver, Solver
    solvers = [Solver(2, n, k=np.exp(synth.uniform(91 + i, (n, n))), precision="fp32_dc", maxit=10)
               for i, n in enumerate(sizes)]
    b = BatchSolver(len(sizes))
    ids = []
    for s in solvers:
        s.set_rhs(synth.uniform_rhs(2, s.n, 95))
        s.set_solution(None)
        ids.append(b.add(s))
    b.step(ids)  # the first step also forms the initial residuals
    before = b.launches()
    b.step(ids)
    return b.launches() - before


@pytest.mark.parametrize("small", [33, 129])
def test_one_outer_residual_launch(small):
    need_gpu()
    # the same levels, so the same launches below the outer step
    assert launches([257, small]) == launches([257, 257])
