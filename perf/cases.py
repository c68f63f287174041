"""What a user of this library has it do, as measurable cases.

A case is a dict of plain values:
  op      "apply", "precondition", "solve", "autograd", "batch" or "paradiag"
  nx, ny, nz   interior points per axis (every n + 1 a power of two; nz = 0: 2D)
  coef    coefficient field of K = -div(a grad .)
  alpha, beta  the shift lambda = alpha + i beta
  precision, tol  plan option and stopping tolerance
  steps   time steps / shifts (batch, paradiag)
Right-hand sides are drawn from the seed on the GPU; the plan (coefficients,
eigenvalue tables, workspace) is what a program keeps between solves.
"""
import math
from types import SimpleNamespace

import torch

import paper_2408_00488_gb300 as csl
from paper_2408_00488_gb300 import autograd as csl_autograd

DEV = "cuda:0"
MAXIT = 2000

# contrast of the fields and the MINRES iterations they take to 1e-8 (the fields
# with a nearly constant coefficient converge in a few steps whatever the size)
ITERATIONS = {"bump": 24, "field": 20, "table2": 14, "exp": 186, "waves": 320}


def _case(op, n, coef="bump", lam=1 + 10j, precision="fp64", tol=1e-8, steps=0, name=None):
    n = tuple(n) + (0,) * (3 - len(n))
    c = dict(op=op, nx=n[0], ny=n[1], nz=n[2], coef=coef, alpha=float(lam.real), beta=float(lam.imag),
             precision=precision, tol=tol, steps=steps)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one operator product on a small grid, as an outer Krylov loop calls it: launch latency
        _case("apply", (63, 63), name="apply_2d_63_fp64"),
        # the absolute-value preconditioner alone (a user's own Krylov method), default precision, 3D
        _case("precondition", (127, 127, 127), "waves", -5 + 50j, name="precondition_3d_127_fp64"),
        # a small solve, default precision: every iteration is launch- and latency-bound
        _case("solve", (63, 63), "bump", 1 + 10j, "fp64", 1e-10, name="solve_2d_63_fp64"),
        # a rectangular domain in the mixed form (FP32 preconditioner, FP64 vectors)
        _case("solve", (511, 255), "exp", 2 + 40j, "fp32_precond", 1e-9, name="solve_2d_511x255_fp32p"),
        # the benchmark's workload in its headline form and in the paper's arithmetic (the default)
        _case("solve", (1023, 1023), "exp", 100j, "fp32", 1e-8, name="solve_2d_1023_fp32"),
        _case("solve", (1023, 1023), "exp", 100j, "fp64", 1e-8, name="solve_2d_1023_fp64"),
        # the 3D benchmark workload
        _case("solve", (127, 127, 127), "waves", -5 + 50j, "fp32", 1e-9, name="solve_3d_127_fp32"),
        # a ragged 3D box with the tensor-core transforms
        _case("solve", (127, 63, 31), "waves", -5 + 50j, "bf16x3", 1e-9, name="solve_3d_127x63x31_bf16x3"),
        # a grid of the paper's Table 2(a): long FP64 lines, few iterations
        _case("solve", (4095, 4095), "table2", -100 + 100j, "fp64", 1e-8, name="solve_2d_4095_fp64"),
        # all shifts of an alpha-circulant time discretisation on three grids, one call
        _case("batch", (511, 511), "bump", 0j, "fp32", 1e-9, 64, name="batch_2d_64_shifts_fp32"),
        # gradients of a misfit with respect to the right-hand side and the coefficient (solve, adjoint, gradient)
        _case("autograd", (511, 511), "field", 1 + 20j, "fp64", 1e-10, name="autograd_2d_511_fp64"),
        # an all-at-once time solve over the batched shifted solves
        _case("paradiag", (127, 127), "bump", 0j, "fp32", 1e-10, 64, name="paradiag_2d_127_64_fp32"),
    ]


def draw(rng):
    size = lambda lo, hi: (1 << rng.randint(lo, hi)) - 1  # noqa: E731
    lam = complex(round(rng.uniform(-5, 50), 2), round(math.exp(rng.uniform(math.log(5), math.log(150))), 2))
    op = rng.choice(["apply", "precondition", "solve", "solve", "solve", "solve", "batch", "autograd", "paradiag"])
    dim = rng.choice([2, 2, 3])
    if op in ("apply", "precondition"):
        n = (size(4, 10), size(4, 10)) if dim == 2 else (size(3, 7), size(3, 7), size(3, 7))
        return _case(op, n, rng.choice(["bump", "exp"]) if dim == 2 else "waves", lam)
    if op == "batch":
        n = size(5, 8)
        return _case(op, (n, n), "bump", 0j, rng.choice(["fp32", "fp64"]), 1e-9, rng.choice([8, 16, 32]))
    if op == "autograd":
        return _case(op, (size(5, 9), size(5, 9)), "bump", lam, "fp64", 1e-10)
    if op == "paradiag":
        n = size(4, 7)
        return _case(op, (n, n), "bump", 0j, rng.choice(["fp32", "fp64"]), 1e-10, rng.choice([16, 32, 64]))
    if dim == 2 and rng.random() < 0.2:  # longer lines, as in the paper's larger tables
        return _case(op, (size(9, 12), size(9, 11)), "table2", lam, "fp64", 1e-8)
    if dim == 2:
        precision = rng.choice(["fp32", "fp32_precond", "fp64"])
        n = (size(4, 10), size(4, 10 if precision != "fp64" else 9))
        return _case(op, n, rng.choice(["bump", "exp"]), lam, precision, 1e-10 if precision == "fp64" else 1e-9)
    precision = rng.choice(["fp32", "fp64", "bf16x3", "bf16x6"])
    n = (size(4, 7), size(4, 6), size(4, 6))
    return _case(op, n, "waves", lam, precision, 1e-10 if precision == "fp64" else 1e-9)


# --- inputs -----------------------------------------------------------------
def _axes(case):
    return [case["nx"], case["ny"]] + ([case["nz"]] if case["nz"] else [])


def _shape(ns):
    return tuple(reversed(ns))


def _coefficient(kind):
    if kind == "bump":
        return lambda *c: 1 + 0.5 * torch.sin(math.pi * c[0]) * torch.sin(math.pi * c[1])
    if kind == "exp":
        return lambda *c: torch.exp(math.log(10.0) * c[0] * c[1])
    if kind == "table2":
        return lambda *c: (20 + c[0] * c[0]) * (20 + c[1] * c[1])
    if kind == "waves":
        return lambda *c: 1 + 0.9 * torch.sin(2 * math.pi * c[0]) * torch.sin(2 * math.pi * c[1]) * torch.sin(
            2 * math.pi * c[2])
    if kind == "field":  # a smooth field of a few modes
        return lambda *c: 1.25 + 0.25 * torch.sin(5.0 * c[0] + 3.0 * c[1] * c[1]) * torch.cos(7.0 * c[1] - 2.0 * c[0])
    raise ValueError(kind)


def _faces(ns, kind):
    """Samples of a at the face midpoints, (x-faces, y-faces[, z-faces])."""
    a, dim, out = _coefficient(kind), len(ns), []
    for axis in range(dim):
        coords, shape = [], []
        for d, n in enumerate(ns):
            h = 1.0 / (n + 1)
            i = torch.arange(n + (d == axis), dtype=torch.float64, device=DEV)
            coords.append(((i + (0.5 if d == axis else 1.0)) * h).reshape([-1 if e == dim - 1 - d else 1
                                                                           for e in range(dim)]))
            shape.append(n + (d == axis))
        out.append(a(*coords).expand(_shape(shape)).contiguous())
    return out


def _complex(shape, gen):
    return torch.view_as_complex(torch.rand(tuple(shape) + (2,), dtype=torch.float64, device=DEV, generator=gen) * 2 - 1)


def _batch_grids(case):
    """The grids of a batch: the case's and its two coarsenings."""
    return [(case["nx"] + 1 >> k) - 1 for k in (2, 1, 0)]


def _shifts(steps, eps=1e-4):
    """Eigenvalues of the alpha-circulant backward-Euler matrix on [0, 1]."""
    w = [complex(math.cos(2 * math.pi * k / steps), math.sin(2 * math.pi * k / steps)) for k in range(steps)]
    return [(1 - eps ** (1.0 / steps) * v) * steps for v in w]


def prepare(case, seed):
    ns = _axes(case)
    shape, lam, op = _shape(ns), complex(case["alpha"], case["beta"]), case["op"]
    gen = torch.Generator(device=DEV).manual_seed(seed)
    s = SimpleNamespace(op=op, tol=case["tol"])
    if op == "batch":
        systems, s.f = [], []
        for n in _batch_grids(case):
            faces = _faces((n, n), case["coef"])
            systems += [(faces, sh) for sh in _shifts(case["steps"])]
            s.f.append(_complex((case["steps"], n, n), gen))
        s.plan = csl.Batch(systems, precision=case["precision"])
        return s
    faces = _faces(ns, case["coef"])
    if op == "paradiag":
        s.u0 = _complex(shape, gen)
        s.g = 0.1 * _complex((case["steps"],) + shape, gen)
        s.plan = csl.ParaDiag(faces, case["steps"], 1.0 / case["steps"], 1e-4, precision=case["precision"])
        return s
    s.f = _complex(shape, gen)
    if op == "autograd":
        s.f.requires_grad_(True)
        s.faces = [a.requires_grad_(True) for a in faces]
        s.d = torch.randn(shape, dtype=torch.float64, device=DEV, generator=gen)
        s.lam, s.precision = lam, case["precision"]
        return s
    s.plan = csl.Plan(faces, lam, precision=case["precision"])
    return s


def run(s):
    if s.op == "apply":
        return s.plan.apply(s.f)
    if s.op == "precondition":
        return s.plan.precondition(s.f)
    if s.op == "solve":
        z, _ = s.plan.solve(s.f, tol=s.tol, maxit=MAXIT)
        return z
    if s.op == "autograd":
        z = csl_autograd.solve(s.f, s.faces, s.lam, tol=s.tol, maxit=MAXIT, precision=s.precision)
        loss = 0.5 * ((z.real - s.d) ** 2).sum()
        grads = torch.autograd.grad(loss, [s.f] + s.faces)
        return {"z": z.detach(), "grad_f": grads[0], "grad_faces": list(grads[1:])}
    if s.op == "batch":
        out = [torch.empty_like(f) for f in s.f]
        s.plan.solve([v for f in s.f for v in f], tol=s.tol, maxit=MAXIT, outs=[v for z in out for v in z])
        return out
    u, _ = s.plan.solve(s.u0, s.g, tol=s.tol, inner_tol=1e-10)
    return u


# --- work -------------------------------------------------------------------
def _transform_flops(ns, points):
    """One separable sine transform of complex points: an FFT of odd data per axis."""
    return points * sum(2.0 * 2.5 * math.log2(2 * (n + 1)) for n in ns)


def work(case):
    ns, op = _axes(case), case["op"]
    points = float(math.prod(ns))
    dim = len(ns)
    faces = 8.0 * dim * points
    if op == "apply":
        return {"bytes": 32 * points + faces, "flops": (8 * dim + 8) * points}
    if op == "precondition":
        return {"bytes": 32 * points, "flops": 2 * _transform_flops(ns, points) + 2 * points}
    its = ITERATIONS[case["coef"]] * math.log(case["tol"]) / math.log(1e-8)

    def solve(ns, points):  # per iteration: operator, P^-1, Lanczos step, update, two inner products
        return its * (2 * _transform_flops(ns, points) + (8 * dim + 34) * points)

    if op == "solve":
        return {"bytes": 32 * points + faces, "flops": solve(ns, points)}
    if op == "autograd":
        return {"bytes": 64 * points + 2 * faces, "flops": 2 * solve(ns, points)}
    if op == "batch":
        grids = _batch_grids(case)
        return {"bytes": sum(case["steps"] * 32.0 * n * n + 16.0 * n * n for n in grids),
                "flops": sum(case["steps"] * solve((n, n), float(n * n)) for n in grids)}
    return {"bytes": (case["steps"] * 32 + 16) * points + faces, "flops": case["steps"] * 3 * solve(ns, points)}


# --- the values in 64 bits ----------------------------------------------------
class _Reference:
    """The operator and a direct constant-coefficient solver with plain torch in
    FP64; vectors carry leading batch dimensions before the grid's."""

    def __init__(self, faces, lam):
        self.dim = len(faces)
        self.ns = [faces[0].shape[-1] - 1] + [faces[0].shape[-1 - d] for d in range(1, self.dim)]
        self.h = [1.0 / (n + 1) for n in self.ns]
        self.faces = [f.detach() / (h * h) for f, h in zip(faces, self.h)]
        self.gamma = math.sqrt(float(min(f.min() for f in faces)) * float(max(f.max() for f in faces)))
        self.lam = torch.as_tensor(lam, dtype=torch.complex128, device=DEV).reshape([-1] + [1] * self.dim)
        mu = 0.0
        for d, (n, h) in enumerate(zip(self.ns, self.h)):
            k = torch.arange(1, n + 1, dtype=torch.float64, device=DEV)
            m = (2.0 / h * torch.sin(0.5 * math.pi * h * k)) ** 2
            mu = mu + m.reshape([-1] + [1] * d)
        self.mu = mu

    def apply(self, z):
        out = self.lam * z
        for d, a in enumerate(self.faces):
            ax = -1 - d
            p = torch.zeros_like(z.narrow(ax, 0, 1))
            flux = a * torch.diff(torch.cat([p, z, p], ax), dim=ax)
            out -= torch.diff(flux, dim=ax)
        return out

    def _sine(self, v):
        for d in range(self.dim):
            ax = -1 - d
            p = torch.zeros_like(v.narrow(ax, 0, 1))
            n = v.shape[ax]
            v = torch.fft.fft(torch.cat([p, v, p, -v.flip(ax)], ax), dim=ax).narrow(ax, 1, n) * 0.5j
            v = v * math.sqrt(2.0 / (n + 1))
        return v

    def constant(self, v, scale):
        return self._sine(self._sine(v) * scale)

    def solve(self, f):
        """(K + lam) z = f by conjugate-orthogonal CG preconditioned with the
        constant-coefficient operator, restarted on the true residual."""
        scale = 1.0 / (self.gamma * self.mu + self.lam)
        dims = tuple(range(-self.dim, 0))
        f = f.reshape((-1,) + tuple(f.shape[-self.dim:]))
        dot = lambda a, b: (a * b).sum(dims, keepdim=True)  # noqa: E731
        norm = lambda a: float((torch.linalg.vector_norm(a, dim=dims) / fn).max())  # noqa: E731
        fn = torch.linalg.vector_norm(f, dim=dims)
        z, best, bad = torch.zeros_like(f), math.inf, 0
        keep = z
        for _ in range(8):
            r = f - self.apply(z)
            now = norm(r)
            if now < best:
                best, keep = now, z.clone()
            if now < 3e-15 or bad:
                break
            v = self.constant(r, scale)
            p, rho = v, dot(r, v)
            target = max(now * 1e-9, 1e-16)
            for it in range(300):
                q = self.apply(p)
                step = rho / dot(p, q)
                z = z + step * p
                r = r - step * q
                if it % 4 == 3 and norm(r) < target:
                    break
                v = self.constant(r, scale)
                new = dot(r, v)
                p = v + (new / rho) * p
                rho = new
            bad = norm(f - self.apply(z)) > 0.5 * now
        return keep


def exact(case, seed):
    with torch.no_grad():
        return _exact(case, seed)


def _exact(case, seed):
    ns = _axes(case)
    shape, lam, op = _shape(ns), complex(case["alpha"], case["beta"]), case["op"]
    gen = torch.Generator(device=DEV).manual_seed(seed)
    if op == "batch":
        out = []
        for n in _batch_grids(case):
            f = _complex((case["steps"], n, n), gen)
            faces, shifts = _faces((n, n), case["coef"]), _shifts(case["steps"])
            out.append(torch.cat([_Reference(faces, shifts[k:k + 16]).solve(f[k:k + 16])
                                  for k in range(0, case["steps"], 16)]))
        return out
    faces = _faces(ns, case["coef"])
    if op == "paradiag":
        u, g = _complex(shape, gen), 0.1 * _complex((case["steps"],) + shape, gen)
        ref, out = _Reference(faces, case["steps"] + 0j), []
        for step in range(case["steps"]):
            u = ref.solve(g[step] + case["steps"] * u)[0]
            out.append(u)
        return torch.stack(out)
    f = _complex(shape, gen)
    ref = _Reference(faces, lam)
    if op == "apply":
        return ref.apply(f[None])[0]
    if op == "precondition":
        return ref.constant(f[None], 1.0 / torch.abs(ref.gamma * ref.mu + ref.lam))[0]
    z = ref.solve(f)[0]
    if op == "solve":
        return z
    d = torch.randn(shape, dtype=torch.float64, device=DEV, generator=gen)
    y = _Reference(faces, lam.conjugate()).solve((z.real - d).to(torch.complex128))[0]
    grads = []
    for axis, h in enumerate(ref.h):
        ax = -1 - axis
        p = torch.zeros_like(z.narrow(ax, 0, 1))
        dz = torch.diff(torch.cat([p, z, p], ax), dim=ax)
        dy = torch.diff(torch.cat([p, y, p], ax), dim=ax)
        grads.append(-(dy.conj() * dz).real / (h * h))
    return {"z": z, "grad_f": y, "grad_faces": grads}
