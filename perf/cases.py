"""Performance cases: the solves this framework is used for, through its public entry points.

Each case is one pass of a user's program that keeps its solver (hierarchy, arena, captured cycles) and has a new
right-hand side on the GPU: hand it over, solve to a relative residual, take the solution into its own device array.
Four families, one per kind of handle the package offers:

  node    Solver       -sum_d c_d u_dd = f, or -div(k grad u) = f, on n = 2^m + 1 nodes per dimension
  batch   BatchSolver  many independent problems of the node family, of uneven sizes, solved together
  cell    CCSolver     sigma u - sum_d c_d u_dd = f on n = 2^m cells per dimension
  cdiff   CDSolver     one implicit Euler step of nonlinear complex diffusion on n x n cells

Sizes and settings are those of bench.py's workloads, of the solve server's defaults and of the tests.
"""
import ctypes
import math

import torch

from paper_1406_5369_gb300 import BatchSolver, CCSolver, CDSolver, Solver, load

MAXIT = 100


# ------------------------------------------------------------------ the cases

def node(name, dim, n, precision, smoother, nu, *, omega=1.0, inner=1, tol=1e-10, maxit=MAXIT, rhs="uniform",
         dirichlet=False, lognormal=0.0, cx=1.0, cy=1.0, cz=1.0):
    c = dict(family="node", dim=dim, n=n, precision=precision, smoother=smoother, omega=omega, nu1=nu[0], nu2=nu[1],
             inner=inner, tol=tol, maxit=maxit, rhs=rhs, dirichlet=dirichlet, lognormal=lognormal, cx=cx, cy=cy, cz=cz)
    return dict(c, name=name) if name else c


def batch(name, dim, count, mlo, mhi, precision, smoother, nu, *, omega=1.0, inner=3, tol=1e-10, lognormal=0.0):
    c = dict(family="batch", dim=dim, count=count, mlo=mlo, mhi=mhi, precision=precision, smoother=smoother,
             omega=omega, nu1=nu[0], nu2=nu[1], inner=inner, tol=tol, maxit=MAXIT, lognormal=lognormal)
    return dict(c, name=name) if name else c


def cell(name, dim, n, bc, smoother, nu, *, omega=1.0, sigma=1.0, tol=1e-8, cx=1.0, cy=1.0, cz=1.0, coarsest=1):
    c = dict(family="cell", dim=dim, n=n, bc=bc, smoother=smoother, omega=omega, nu1=nu[0], nu2=nu[1], sigma=sigma,
             tol=tol, cx=cx, cy=cy, cz=cz, coarsest=coarsest)
    return dict(c, name=name) if name else c


def cdiff(name, n, smoother, nu, *, omega=1.0, tau=1e-4, theta=math.pi / 30, kappa=0.1, tol=1e-8):
    c = dict(family="cdiff", n=n, smoother=smoother, omega=omega, nu1=nu[0], nu2=nu[1], tau=tau, theta=theta,
             kappa=kappa, tol=tol)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the paper's own small problem: ten FP64 V(2,1) cycles on 129^2, a smooth right-hand side; launches and
        # latency are all of it
        node("node2d_129_fp64", 2, 129, "fp64", "rbgs", (2, 1), tol=0.0, maxit=10, rhs="smooth"),
        # one ordinary request of the solve server, alone on the GPU
        node("node2d_513_fp32dc", 2, 513, "fp32_dc", "rbgs", (2, 1), inner=3),
        # the headline: a large 2D Poisson problem to 1e-10 by FP32 inner cycles in FP64 defect correction
        node("node2d_8193_fp32dc", 2, 8193, "fp32_dc", "rbgs", (2, 1), inner=3),
        # Table 2 of the paper, double precision: a program that wants every operation in FP64
        node("node2d_4097_fp64_rbgs", 2, 4097, "fp64", "rbgs", (2, 2), tol=1e-8),
        node("node2d_4097_fp64_jacobi", 2, 4097, "fp64", "jacobi", (2, 2), omega=0.8, tol=1e-8),
        node("node3d_257_fp64_rbgs", 3, 257, "fp64", "rbgs", (2, 2), tol=1e-8, dirichlet=True),
        # the large 3D problem: BF16-stored Jacobi cycles in FP64 defect correction, white noise on the right
        node("node3d_513_bf16dc", 3, 513, "bf16_dc", "jacobi", (2, 2), omega=6.0 / 7.0, inner=3, rhs="normal"),
        # many small uneven problems with variable coefficients (porous media samples), one batch
        batch("batch2d_lognormal_128", 2, 128, 5, 10, "fp32_dc", "rbgs", (2, 1), tol=1e-8, lognormal=1.0),
        # the 3D share of the solve server's load: uneven sizes, its default settings
        batch("batch3d_server_24", 3, 24, 5, 8, "bf16_dc", "jacobi", (2, 2), omega=6.0 / 7.0),
        # implicit diffusion steps on cell-centred grids at Table 2's sizes: zero-flux 2D, fixed-value 3D
        cell("cell2d_4096_neumann", 2, 4096, "neumann", "rbgs", (2, 2)),
        cell("cell3d_128_dirichlet", 3, 128, "dirichlet", "rbgs", (2, 2), sigma=100.0),
        # one denoising step of a photograph-sized image
        cdiff("cdiff_2048", 2048, "jacobi", (2, 2), omega=0.8),
    ]


def draw(rng):
    family = rng.choice(("node", "node", "node", "node", "batch", "cell", "cell", "cdiff"))
    nu = rng.choice(((2, 1), (2, 2), (1, 2), (3, 2), (2, 3)))
    if family == "node":
        dim = rng.choice((2, 2, 3))
        precision = rng.choice(("fp64", "fp32_dc") if dim == 2 else ("fp64", "fp32_dc", "bf16_dc"))
        smoother = rng.choice(("rbgs", "rbgs", "jacobi"))
        # the tops keep a drawn pass below the longest listed one
        top = {(2, "fp64"): 11, (2, "fp32_dc"): 13 if smoother == "rbgs" else 12, (3, "fp64"): 7}.get((dim, precision), 8)
        m = rng.randint(5 if dim == 2 else 4, top)
        kind = rng.choice(("poisson", "poisson", "anisotropic") + (("lognormal",) if dim == 2 else ()))
        if kind == "lognormal":  # the answer in 64 bits of a larger one would take over twenty seconds
            m = min(m, 11)
        omega = rng.choice((1.0, round(rng.uniform(0.95, 1.15), 3)))
        if smoother == "jacobi":
            omega = round(rng.uniform(0.75, 0.85), 3) if dim == 2 else round(rng.uniform(0.8, 6.0 / 7.0), 3)
            nu = rng.choice(((2, 2), (2, 1), (3, 3)))
        c = [round(rng.uniform(0.7, 1.4), 3) for _ in range(3)] if kind == "anisotropic" else [1.0] * 3
        return node(None, dim, (1 << m) + 1, precision, smoother, nu, omega=omega,
                    inner=rng.randint(1, 3) if precision != "fp64" else 1,
                    tol=1e-10 if precision == "bf16_dc" else 10.0 ** -rng.randint(8, 10),
                    rhs=rng.choice(("uniform", "normal", "smooth")), dirichlet=rng.random() < 0.4,
                    lognormal=round(rng.uniform(0.5, 1.0), 3) if kind == "lognormal" else 0.0,
                    cx=c[0], cy=c[1], cz=c[2])
    if family == "batch":
        if rng.random() < 0.5:
            mlo = rng.randint(4, 5)
            return batch(None, 3, rng.randint(3, 24), mlo, rng.randint(mlo + 1, 7), "bf16_dc", "jacobi", (2, 2),
                         omega=round(rng.uniform(0.8, 6.0 / 7.0), 3))
        mlo = rng.randint(5, 7)
        lognormal = rng.choice((0.0, round(rng.uniform(0.5, 1.0), 3)))
        mhi = rng.randint(mlo, 10)
        nodes = sum(4 ** m for m in range(mlo, mhi + 1)) / (mhi - mlo + 1)
        most = max(4, min(160, int(30e6 / nodes)))
        return batch(None, 2, int(round(math.exp(rng.uniform(math.log(4), math.log(most))))), mlo, mhi, "fp32_dc",
                     "rbgs", (2, 1), omega=rng.choice((1.0, round(rng.uniform(1.0, 1.15), 3))),
                     inner=rng.randint(1, 3), tol=1e-8 if lognormal else 1e-10, lognormal=lognormal)
    if family == "cell":
        dim = rng.choice((2, 2, 3))
        # Jacobi converges on these transfers with zero-flux faces in 2D only
        smoother = rng.choice(("rbgs", "rbgs", "jacobi")) if dim == 2 else "rbgs"
        bc = "neumann" if smoother == "jacobi" else rng.choice(("neumann", "neumann", "dirichlet"))
        m = rng.randint(5, 12 if (bc, smoother) == ("neumann", "rbgs") else 11) if dim == 2 else rng.randint(4, 7)
        anisotropic = smoother == "rbgs" and rng.random() < 0.3
        c = [round(rng.uniform(0.8, 1.25), 3) for _ in range(3)] if anisotropic else [1.0] * 3
        return cell(None, dim, 1 << m, bc, smoother, (2, 2), omega=1.0 if smoother == "rbgs" else 0.8,
                    sigma=round(math.exp(rng.uniform(0.0, math.log(1000.0))), 3), cx=c[0], cy=c[1], cz=c[2],
                    tol=10.0 ** -rng.randint(6, 9), coarsest=rng.choice((1, 1, 2, 4)))
    smoother = rng.choice(("rbgs", "jacobi"))
    return cdiff(None, 1 << rng.randint(6, 11), smoother, rng.choice(((2, 2), (2, 1))),
                 omega=1.0 if smoother == "rbgs" else 0.8, tau=round(10.0 ** rng.uniform(-5, -3), 7),
                 kappa=round(rng.uniform(0.08, 0.3), 3), tol=10.0 ** -rng.randint(6, 9))


# ------------------------------------------------------------------ inputs

def generator(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + salt)
    return g


def modes(shape, g):
    """A few random low sine modes, zero on the boundary of the unit cube."""
    x = [torch.linspace(0.0, 1.0, s, dtype=torch.float64, device="cuda") for s in shape]
    out = torch.zeros(shape, dtype=torch.float64, device="cuda")
    a = torch.randn(4, generator=g, dtype=torch.float64, device="cuda")
    for q in range(4):
        term = a[q] * torch.ones((1,) * len(shape), dtype=torch.float64, device="cuda")
        for d in range(len(shape)):
            view = [1] * len(shape)
            view[d] = -1
            term = term * torch.sin((1 + (q + d) % 3) * math.pi * x[d]).view(view)
        out += term
    return out


def right_side(dim, n, kind, g):
    shape = (n,) * dim
    if kind == "normal":
        return torch.randn(shape, generator=g, dtype=torch.float64, device="cuda")
    if kind == "smooth":
        return 20.0 * modes(shape, g)
    return 2.0 * torch.rand(shape, generator=g, dtype=torch.float64, device="cuda") - 1.0


def boundary_values(dim, n, g):
    """A smooth field whose boundary nodes are the Dirichlet values."""
    x = torch.linspace(0.0, 1.0, n, dtype=torch.float64, device="cuda")
    a = torch.rand(2 * dim, generator=g, dtype=torch.float64, device="cuda") * 0.02
    out = torch.zeros((n,) * dim, dtype=torch.float64, device="cuda")
    for d in range(dim):
        view = [1] * dim
        view[d] = -1
        out = out + (a[2 * d] * torch.cos(math.pi * x) + a[2 * d + 1] * x * x).view(view)
    return out


def diffusivity(dim, n, sigma, g):
    return torch.exp(sigma * torch.randn((n,) * dim, generator=g, dtype=torch.float64, device="cuda"))


def node_inputs(case, seed):
    g = generator(seed)
    dim, n = case["dim"], case["n"]
    f = right_side(dim, n, case["rhs"], g)
    k = diffusivity(dim, n, case["lognormal"], g) if case["lognormal"] else None
    b = boundary_values(dim, n, g) if case["dirichlet"] else None
    return f, k, b


def batch_sizes(case):
    """The problems' sizes: every 2^m + 1 of the range, dealt out in turn."""
    return [(1 << (case["mlo"] + p % (case["mhi"] - case["mlo"] + 1))) + 1 for p in range(case["count"])]


def batch_inputs(case, seed):
    out = []
    for p, n in enumerate(batch_sizes(case)):
        g = generator(seed, 7 + p)
        f = right_side(case["dim"], n, "uniform", g)
        out.append((f, diffusivity(case["dim"], n, case["lognormal"], g) if case["lognormal"] else None))
    return out


def cell_inputs(case, seed):
    """A noisy field that one implicit Euler step smooths: f = sigma u0."""
    g = generator(seed)
    return case["sigma"] * right_side(case["dim"], case["n"], "uniform", g)


def image(case, seed):
    """A bump with noise; the imaginary part is what earlier steps left there."""
    g, n = generator(seed), case["n"]
    x = (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / n
    c = torch.rand(2, generator=g, dtype=torch.float64, device="cuda") * 0.4 + 0.3
    bump = torch.exp(-((x[None, :] - c[0]) ** 2 + (x[:, None] - c[1]) ** 2) / 0.05)
    re = bump + 0.3 * (2.0 * torch.rand((n, n), generator=g, dtype=torch.float64, device="cuda") - 1.0)
    im = 0.02 * (2.0 * torch.rand((n, n), generator=g, dtype=torch.float64, device="cuda") - 1.0)
    return torch.complex(re, im)


# ------------------------------------------------------------------ one pass

def prepare(case, seed):
    st = {"case": case}
    if case["family"] == "node":
        f, k, b = node_inputs(case, seed)
        st["f"] = f
        st["solver"] = Solver(case["dim"], case["n"], stencil=(case["cx"], case["cy"], case["cz"]), k=k, dirichlet=b,
                              smoother=case["smoother"], omega=case["omega"], nu1=case["nu1"], nu2=case["nu2"],
                              maxit=case["maxit"], precision=case["precision"], inner_cycles=case["inner"])
        st["u"] = torch.empty_like(f)
    elif case["family"] == "batch":
        inputs = batch_inputs(case, seed)
        st["f"] = [f for f, _ in inputs]
        st["solvers"] = [Solver(case["dim"], f.shape[0], k=k, smoother=case["smoother"], omega=case["omega"],
                                nu1=case["nu1"], nu2=case["nu2"], maxit=case["maxit"], precision=case["precision"],
                                inner_cycles=case["inner"]) for f, k in inputs]
        st["batch"] = BatchSolver(case["count"])
        st["u"] = torch.empty(sum(f.numel() for f in st["f"]), dtype=torch.float64, device="cuda")
        parts = torch.split(st["u"], [f.numel() for f in st["f"]])
        st["parts"] = [p.view(f.shape) for p, f in zip(parts, st["f"])]
    elif case["family"] == "cell":
        st["f"] = cell_inputs(case, seed)
        st["solver"] = CCSolver(case["dim"], case["n"], c=(case["cx"], case["cy"], case["cz"]), sigma=case["sigma"],
                                bc=case["bc"], smoother=case["smoother"], omega=case["omega"], nu1=case["nu1"],
                                nu2=case["nu2"], coarsest_n=case["coarsest"], maxit=MAXIT)
        st["start"] = torch.zeros_like(st["f"])
        st["u"] = torch.empty_like(st["f"])
    else:
        st["f"] = image(case, seed)
        st["solver"] = CDSolver(case["n"], tau=case["tau"], theta=case["theta"], kappa=case["kappa"],
                                smoother=case["smoother"], omega=case["omega"], nu1=case["nu1"], nu2=case["nu2"],
                                maxit=MAXIT)
        st["u"] = torch.empty_like(st["f"])
    return st


def device_field(get_field, ctx, out):
    """Level 0's u into a device array, through the C interface (the Python handles' get_field is for host arrays)."""
    status = get_field(ctx, 0, 0, ctypes.c_void_p(out.data_ptr()))
    if status != 0:
        raise RuntimeError(load().mg_last_error().decode())


def run(st):
    case = st["case"]
    if case["family"] == "node":
        s = st["solver"]
        s.set_rhs(st["f"])
        s.set_solution(None)
        cycles, _, _ = s.solve(case["tol"], raise_on_noconv=case["tol"] > 0.0)
        return {"u": s.get_solution(st["u"]), "cycles": cycles}
    if case["family"] == "batch":
        b, ids = st["batch"], []
        for s, f in zip(st["solvers"], st["f"]):
            s.set_rhs(f)
            s.set_solution(None)
            ids.append(b.add(s))
        steps, _ = b.solve(case["tol"], maxit=case["maxit"])
        for s, i, u in zip(st["solvers"], ids, st["parts"]):
            s.get_solution(u)
            b.remove(i)
        return {"u": st["u"], "steps": steps[ids]}
    s = st["solver"]
    if case["family"] == "cell":
        s.set_rhs(st["f"])
        s.set_solution(st["start"])
        cycles, _, _ = s.solve(case["tol"])
        device_field(load().mg_cc_get_field, s.ctx, st["u"])
    else:
        cycles, _, _ = s.time_step(st["f"], case["tol"])
        device_field(load().mg_cd_get_field, s.ctx, st["u"])
    return {"u": st["u"], "cycles": cycles}


def work(case):
    """Bytes: the right-hand side (and coefficients) read once and the solution written once. Operations: the V-cycles
    a method of this kind needs for the tolerance (a factor of about ten each), one multiplication and addition per
    stencil entry, point and sweep."""
    dim = 2 if case["family"] == "cdiff" else case["dim"]
    points = (sum(n ** dim for n in batch_sizes(case)) if case["family"] == "batch" else case["n"] ** dim)
    cycles = case["maxit"] if case["tol"] == 0.0 else math.ceil(-math.log10(case["tol"]))
    per_cycle = (case["nu1"] + case["nu2"] + 1) * 2 * (2 * dim + 1) * (4.0 / 3.0 if dim == 2 else 8.0 / 7.0)
    word = 16 if case["family"] == "cdiff" else 8
    return {"bytes": points * word * (3 if case.get("lognormal") else 2),
            "flops": points * cycles * per_cycle * (4 if case["family"] == "cdiff" else 1)}


# ------------------------------------------------------------------ the answers in 64 bits
# Constant coefficients: the discrete problem is diagonal in sine or cosine modes. Variable coefficients: conjugate
# gradients in FP64, preconditioned with the constant-coefficient solution.

def along(x, d, op):
    """op along the last axis, applied to axis d."""
    return op(x.transpose(d, -1)).transpose(d, -1)


def dst1(x):
    """2 sum_j x_j sin(pi (j+1)(k+1)/(N+1)) along the last axis; twice gives 2(N+1) x."""
    zero = torch.zeros_like(x[..., :1])
    return -torch.fft.rfft(torch.cat((zero, x, zero, -x.flip(-1)), -1)).imag[..., 1:x.shape[-1] + 1]


def phase(n, sign):
    a = math.pi * torch.arange(n + 1, dtype=torch.float64, device="cuda") / (2 * n)
    return torch.complex(torch.cos(a), sign * torch.sin(a))


def to_modes(x, bc):
    """Cell-centred cosine (zero flux) or sine (fixed value) coefficients along the last axis."""
    n = x.shape[-1]
    if bc == "neumann":
        return (torch.fft.rfft(torch.cat((x, x.flip(-1)), -1)) * phase(n, -1.0)).real[..., :n]
    return (1j * torch.fft.rfft(torch.cat((x, -x.flip(-1)), -1)) * phase(n, -1.0)).real[..., 1:]


def from_modes(c, bc):
    n = c.shape[-1]
    zero = torch.zeros_like(c[..., :1])
    if bc == "neumann":
        y = torch.cat((c, zero), -1) * phase(n, 1.0)
    else:
        y = -1j * torch.cat((zero, c), -1) * phase(n, 1.0)
    return torch.fft.irfft(y, n=2 * n)[..., :n]


def eigenvalues(dim, n, c, count, first):
    """sum_d c_d (4/h^2) sin^2(pi k h / 2), h = 1/n, k = first .. first + count - 1; axis 0 is the slowest."""
    k = torch.arange(first, first + count, dtype=torch.float64, device="cuda")
    one = 4.0 * n * n * torch.sin(math.pi * k / (2 * n)) ** 2
    lam = 0.0
    for d in range(dim):
        view = [1] * dim
        view[dim - 1 - d] = -1
        lam = lam + c[d] * one.view(view)
    return lam


def poisson_modes(f, dim, n, c):
    """The solution on the inner nodes of n per dimension, zero on the boundary; leading axes are a batch."""
    for d in range(-dim, 0):
        f = along(f, d, dst1)
    f = f / eigenvalues(dim, n - 1, c, n - 2, 1) / (2.0 * (n - 1)) ** dim
    for d in range(-dim, 0):
        f = along(f, d, dst1)
    return f


def faces(k, dim, d):
    """Harmonic means of neighbouring nodes along spatial axis d (0 the fastest), on inner rows of the other axes."""
    k = inner_but(k, dim, d)
    lo, hi = k.narrow(-1 - d, 0, k.shape[-1 - d] - 1), k.narrow(-1 - d, 1, k.shape[-1 - d] - 1)
    return 2.0 * lo * hi / (lo + hi)


def inner_but(v, dim, d):
    """Every spatial axis but d without its end nodes (d None: every one)."""
    for a in range(dim):
        if a != d:
            v = v.narrow(-1 - a, 1, v.shape[-1 - a] - 2)
    return v


def node_exact(case, f, k, b):
    """Solutions of a stack of problems of one size (leading axis)."""
    dim, n = case["dim"], f.shape[-1]
    c = (case.get("cx", 1.0), case.get("cy", 1.0), case.get("cz", 1.0))
    ih2 = float(n - 1) ** 2
    u = torch.zeros_like(f)
    if b is not None:
        u += b
        inner_but(u, dim, None).zero_()
    kf = [c[d] * faces(k, dim, d) if k is not None else c[d] for d in range(dim)]

    def apply(v):
        """A v at the inner nodes of full grids v."""
        out = torch.zeros_like(inner_but(v, dim, None))
        for d in range(dim):
            w = inner_but(v, dim, d)
            flux = kf[d] * (w.narrow(-1 - d, 1, n - 1) - w.narrow(-1 - d, 0, n - 1))
            out -= ih2 * (flux.narrow(-1 - d, 1, n - 2) - flux.narrow(-1 - d, 0, n - 2))
        return out

    def dot(v, w):
        return torch.sum(v * w, tuple(range(-dim, 0)), keepdim=True)

    r = inner_but(f, dim, None) - apply(u) if b is not None else inner_but(f, dim, None).clone()
    if k is None:
        inner_but(u, dim, None).copy_(poisson_modes(r, dim, n, c))
        return u
    full = torch.zeros_like(f)
    x = torch.zeros_like(r)
    z = poisson_modes(r, dim, n, c)
    p, rz, stop = z.clone(), dot(r, z), 1e-26 * dot(r, r)
    for _ in range(2000):
        inner_but(full, dim, None).copy_(p)
        q = apply(full)
        a = rz / dot(p, q)
        x += a * p
        r -= a * q
        if bool((dot(r, r) <= stop).all()):
            break
        z = poisson_modes(r, dim, n, c)
        new = dot(r, z)
        p = z + (new / rz) * p
        rz = new
    inner_but(u, dim, None).copy_(x)
    return u


def cell_exact(case, f):
    dim, n, bc = case["dim"], case["n"], case["bc"]
    for d in range(dim):
        f = along(f, d, lambda x: to_modes(x, bc))
    c = (case["cx"], case["cy"], case["cz"])
    f = f / (case["sigma"] + eigenvalues(dim, n, c, n, 0 if bc == "neumann" else 1))
    for d in range(dim):
        f = along(f, d, lambda x: from_modes(x, bc))
    return f


def cdiff_exact(case, un):
    """(1 + tau h^-2 sum g (u_p - u_q)) u = u^n: conjugate gradients for complex symmetric systems."""
    n, s = case["n"], case["tau"] * case["n"] ** 2
    w = 1.0 / (1.0 + (un.imag / (case["kappa"] * case["theta"])) ** 2)
    g = w * complex(math.cos(case["theta"]), math.sin(case["theta"]))
    gx, gy = 0.5 * (g[:, 1:] + g[:, :-1]), 0.5 * (g[1:] + g[:-1])
    mean = case["tau"] * 0.5 * (gx.mean() + gy.mean())
    lam = eigenvalues(2, n, (1.0, 1.0), n, 0)

    def apply(v):
        out = v.clone()
        fx, fy = s * gx * (v[:, 1:] - v[:, :-1]), s * gy * (v[1:] - v[:-1])
        out[:, :-1] -= fx
        out[:, 1:] += fx
        out[:-1] -= fy
        out[1:] += fy
        return out

    def both(v, op):
        return torch.complex(op(v.real), op(v.imag))

    def precondition(v):
        for d in range(2):
            v = both(v, lambda x: along(x, d, lambda y: to_modes(y, "neumann")))
        v = v / (1.0 + mean * lam)
        for d in range(2):
            v = both(v, lambda x: along(x, d, lambda y: from_modes(y, "neumann")))
        return v

    x = precondition(un)
    r = un - apply(x)
    z = precondition(r)
    p, rz, stop = z.clone(), torch.sum(r * z), 1e-14 * torch.linalg.norm(un)
    for _ in range(300):
        if torch.linalg.norm(r) <= stop:
            break
        q = apply(p)
        a = rz / torch.sum(p * q)
        x = x + a * p
        r = r - a * q
        z = precondition(r)
        new = torch.sum(r * z)
        p = z + (new / rz) * p
        rz = new
    return x


def batch_exact(case, seed):
    """Problems of one size stacked, a few million nodes at a time."""
    inputs = batch_inputs(case, seed)
    out = [None] * len(inputs)
    for n in sorted(set(batch_sizes(case))):
        same = [i for i, (f, _) in enumerate(inputs) if f.shape[0] == n]
        most = max(1, 30_000_000 // n ** case["dim"])
        for at in range(0, len(same), most):
            some = same[at:at + most]
            f = torch.stack([inputs[i][0] for i in some])
            k = torch.stack([inputs[i][1] for i in some]) if case["lognormal"] else None
            for i, u in zip(some, node_exact(case, f, k, None)):
                out[i] = u.reshape(-1)
    return torch.cat(out)


def exact(case, seed):
    if case["family"] == "node":
        f, k, b = (x[None] if x is not None else None for x in node_inputs(case, seed))
        u = node_exact(case, f, k, b)[0]
    elif case["family"] == "batch":
        return {"u": batch_exact(case, seed), "steps": None}
    elif case["family"] == "cell":
        u = cell_exact(case, cell_inputs(case, seed))
    else:
        u = cdiff_exact(case, image(case, seed))
    return {"u": u, "cycles": None}
