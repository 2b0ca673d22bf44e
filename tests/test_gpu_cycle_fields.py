"""The fields that V-cycles leave on every level (u, f and r, the residual after
pre-smoothing) are those of Algorithm 1 run one operator at a time, whichever
kernels the cycle took, and reading them changes nothing.

Tolerances: u to 1e-12 of the finest one (which it corrects), f of a coarse level
and r, which are differences, to 1e-12 of diag times the largest u of the level
they come from: some thousand times the rounding of the few dozen operations
behind each value.
The coarse fields have to be of the finest one's order for that: one cycle from a
random start, or three with sweeps weak enough (omega = 0.3) to leave an error.
"""
import numpy as np
import pytest

import synth
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def plain_cycle(s, nu1, nu2, l=0, zero=None):
    """Algorithm 1 by the level operators."""
    if l == s.levels - 1:
        s.coarse_solve()
        return
    s.smooth(l, nu1)
    s.residual(l)
    s.restrict(l)
    s.set_field(l + 1, "u", np.zeros_like(s.get_field(l + 1, "u")))
    plain_cycle(s, nu1, nu2, l + 1)
    s.prolongate(l)
    s.smooth(l, nu2)


def compare(s, ref, diag, order):
    top = s.get_field(0, "u")
    for l, name in order:
        got, want = s.get_field(l, name), ref.get_field(l, name)
        scale = np.abs(ref.get_field(0, "u")).max()
        if name != "u":
            scale = max(diag(max(l - 1, 0)) * np.abs(ref.get_field(max(l - 1, 0), "u")).max(), np.abs(want).max())
        assert np.abs(got - want).max() <= 1e-12 * scale, (l, name)
    assert np.array_equal(s.get_field(0, "u"), top)


def every(levels):
    """r of a middle level first, then everything."""
    return [(levels // 2, "r")] + [(l, name) for l in range(levels) for name in ("r", "f", "u")]


@pytest.mark.parametrize("dim,n,bc,smoother,omega,nu,nc", [
    (2, 8, "neumann", "rbgs", 1.0, (2, 1), 1),
    (2, 64, "neumann", "jacobi", 0.8, (2, 1), 2),
    (2, 128, "dirichlet", "rbgs", 1.1, (2, 2), 1),
    (2, 128, "neumann", "rbgs", 1.0, (0, 2), 4),
    (2, 512, "neumann", "rbgs", 1.0, (2, 2), 1),
    (2, 256, "dirichlet", "jacobi", 0.8, (3, 3), 2),
    (2, 256, "neumann", "rbgs", 1.0, (2, 0), 1),
    (3, 4, "dirichlet", "rbgs", 1.0, (2, 2), 2),
    (3, 8, "neumann", "jacobi", 0.8, (1, 2), 1),
    (3, 32, "neumann", "rbgs", 1.0, (2, 2), 1),
    (3, 64, "dirichlet", "jacobi", 0.8, (0, 3), 4),
    (3, 64, "dirichlet", "rbgs", 1.2, (3, 0), 1),
])
@pytest.mark.parametrize("solve", [False, True])
def test_cell_centred(dim, n, bc, smoother, omega, nu, nc, solve):
    need_gpu()
    from paper_1406_5369_gb300 import CCSolver
    f, u0 = synth.uniform(81, (n,) * dim), synth.uniform(82, (n,) * dim)
    kw = dict(sigma=3.0, bc=bc, smoother=smoother, omega=0.3 if solve else omega, nu1=nu[0], nu2=nu[1], coarsest_n=nc,
              maxit=3)
    s, ref = CCSolver(dim, n, **kw), CCSolver(dim, n, **kw)
    for t in (s, ref):
        t.set_rhs(f)
        t.set_solution(u0)
    if solve:  # three steps, the last one a replayed graph
        s.solve(0.0, raise_on_noconv=False)
    else:
        s.vcycle()
    for _ in range(3 if solve else 1):
        plain_cycle(ref, *nu)
    compare(s, ref, lambda l: 4.0 * dim * (n >> l) ** 2, every(s.levels))


def test_cell_centred_level_calls_after_a_cycle():
    """Level operators and norms work on the fields that the cycle leaves."""
    need_gpu()
    from paper_1406_5369_gb300 import CCSolver
    n = 256
    f = synth.uniform(83, (n, n))
    for call in (lambda t: t.restrict(0), lambda t: t.prolongate(1), lambda t: t.smooth(2, 1), lambda t: t.residual(3),
                 lambda t: t.set_field(2, "u", np.ones((n // 4, n // 4))), lambda t: t.coarse_solve()):
        s, ref = CCSolver(2, n), CCSolver(2, n)
        for t in (s, ref):
            t.set_rhs(f)
            t.set_solution(None)
        s.vcycle()
        plain_cycle(ref, 2, 1)
        call(s)
        call(ref)
        compare(s, ref, lambda l: 8.0 * (n >> l) ** 2, every(s.levels))
        assert abs(s.residual_norm(2) - ref.residual_norm(2)) <= 1e-10 * ref.residual_norm(0)


def cd_pair(n, **kw):
    need_gpu()
    from paper_1406_5369_gb300 import CDSolver
    un = synth.uniform(84, (n, n)) + 0.05j * synth.uniform(85, (n, n))
    s, ref = CDSolver(n, tau=1e-2, **kw), CDSolver(n, tau=1e-2, **kw)
    for t in (s, ref):
        t.begin_step(un)
    return s, ref


@pytest.mark.parametrize("n,smoother,omega,nu", [
    (2, "rbgs", 1.0, (2, 2)),
    (64, "rbgs", 1.0, (2, 2)),
    (128, "jacobi", 0.8, (2, 1)),
    (256, "jacobi", 0.8, (0, 2)),
    (256, "rbgs", 1.2, (3, 0)),
])
@pytest.mark.parametrize("solve", [False, True])
@pytest.mark.parametrize("face_first", [False, True])
def test_complex_diffusion(n, smoother, omega, nu, solve, face_first):
    s, ref = cd_pair(n, smoother=smoother, omega=0.3 if solve else omega, nu1=nu[0], nu2=nu[1], maxit=3)
    if solve:
        s.solve(0.0, raise_on_noconv=False)
    else:
        s.vcycle()
    for _ in range(3 if solve else 1):
        plain_cycle(ref, *nu)
    if face_first:
        assert np.array_equal(s.get_field(0, "gx"), ref.get_field(0, "gx"))
    compare(s, ref, lambda l: 1.0 + 4e-2 * (n >> l) ** 2, every(s.levels))


def test_complex_diffusion_faces_and_norms_leave_the_cycles_as_they_are():
    s, ref = cd_pair(128)
    for t in (s, ref):
        t.vcycle()
    for l in range(s.levels):
        for name in ("gx", "gy"):
            s.get_field(l, name)
        s.residual_norm(l)
    for t in (s, ref):
        t.vcycle()
    assert np.array_equal(s.get_field(0, "u"), ref.get_field(0, "u"))  # the same kernels still
    # the faces are the same on either kind of context, and so are the norms
    norms = [s.residual_norm(l) for l in range(s.levels)]
    faces = [s.get_field(l, name) for l in range(s.levels) for name in ("gx", "gy")]
    s.residual(0)
    assert all(abs(s.residual_norm(l) - v) <= 1e-12 * norms[0] for l, v in enumerate(norms))
    assert all(np.array_equal(a, s.get_field(l, name))
               for a, (l, name) in zip(faces, [(l, name) for l in range(s.levels) for name in ("gx", "gy")]))


def test_complex_diffusion_residual_before_any_cycle():
    s, ref = cd_pair(64)
    ref.residual(0)
    r = s.get_field(0, "r")
    assert np.abs(r - ref.get_field(0, "r")).max() <= 1e-13 * 170
    s.restrict(0)
    ref.restrict(0)
    assert np.abs(s.get_field(1, "f") - ref.get_field(1, "f")).max() <= 1e-13 * 170


# FP64 node grids: the levels above 33 (9 in 3D), whose fields cycles of one kernel
# per operator or the fused FP64 passes leave; red-black 2D passes form no r
@pytest.mark.parametrize("dim,n,smoother,omega,nu,kw", [
    (2, 65, "rbgs", 1.0, (2, 1), {}),
    (2, 129, "rbgs", 1.0, (2, 1), {}),
    (2, 129, "jacobi", 0.8, (1, 2), {}),
    (2, 257, "rbgs", 1.0, (2, 2), dict(cluster_max_n=257)),
    (2, 513, "rbgs", 1.0, (3, 2), {}),
    (2, 513, "jacobi", 0.8, (2, 1), {}),
    (2, 257, "jacobi", 0.8, (3, 3), dict(cluster_max_n=33)),
    (3, 257, "rbgs", 1.0, (1, 2), {}),
    (3, 257, "jacobi", 0.8, (2, 1), {}),
])
@pytest.mark.parametrize("solve", [False, True])
def test_node_fp64(dim, n, smoother, omega, nu, kw, solve):
    need_gpu()
    from paper_1406_5369_gb300 import Solver
    f, b = synth.uniform(86, (n,) * dim), synth.uniform(87, (n,) * dim)
    u0 = synth.uniform(88, (n,) * dim)
    kw = dict(kw, smoother=smoother, omega=0.3 if solve else omega, nu1=nu[0], nu2=nu[1], maxit=3, dirichlet=b)
    s, ref = Solver(dim, n, **kw), Solver(dim, n, fuse=False, **kw)
    for t in (s, ref):
        t.set_rhs(f)
        t.set_solution(u0)
        if solve:
            t.solve(0.0, raise_on_noconv=False)
        else:
            t.vcycle()
    top = 33 if dim == 2 else 9
    names = ("f", "u") if smoother == "rbgs" and dim == 2 else ("r", "f", "u")
    order = [(l, name) for l in range(s.levels) if s.level_size(l) > top for name in names]
    compare(s, ref, lambda l: 2.0 * dim * (n >> l) ** 2, order[::-1] + order)


def test_node_fp64_residual_of_the_caller():
    """Fused red-black cycles leave r as the caller's mg_residual left it."""
    need_gpu()
    from paper_1406_5369_gb300 import Solver
    for n in (65, 129, 513):
        s = Solver(2, n)
        s.set_rhs(synth.uniform_rhs(2, n, 89))
        s.residual(0)
        r = s.get_field(0, "r")
        s.vcycle()
        s.get_field(1, "u")
        assert np.array_equal(s.get_field(0, "r"), r)


def test_node_fp64_batch_after_a_cycle():
    """A context that has run a cycle of its own joins a batch with every field in place."""
    need_gpu()
    from paper_1406_5369_gb300 import BatchSolver, Solver
    n = 257
    f = synth.uniform_rhs(2, n, 90)
    got = []
    for own in (True, False):
        s = Solver(2, n, smoother="jacobi", omega=0.8, nu1=2, nu2=2)
        s.set_rhs(f)
        s.vcycle() if own else None
        s.set_solution(None)
        b = BatchSolver(1)
        b.add(s)
        b.solve(1e-8, maxit=50)
        got.append(s.get_solution())
    assert np.array_equal(got[0], got[1])


@pytest.mark.parametrize("n,nu", [(65, (2, 0)), (129, (3, 2)), (513, (3, 2)), (257, (1, 4))])
def test_node_fp64_red_black_without_fused_passes(n, nu):
    """Red-black cycles with no or more than two sweeps a phase form r on every level above 33."""
    need_gpu()
    from paper_1406_5369_gb300 import Solver
    f, u0 = synth.uniform_rhs(2, n, 86), synth.uniform(88, (n, n))
    u0[0], u0[-1], u0[:, 0], u0[:, -1] = 0, 0, 0, 0
    kw = dict(nu1=nu[0], nu2=nu[1])
    s, ref = Solver(2, n, **kw), Solver(2, n, fuse=False, **kw)
    for t in (s, ref):
        t.set_rhs(f)
        t.set_solution(u0)
        t.vcycle()
    order = [(l, name) for l in range(s.levels) if s.level_size(l) > 33 for name in ("r", "f", "u")]
    compare(s, ref, lambda l: 4.0 * (n >> l) ** 2, order)
