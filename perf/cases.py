"""The work that users of the library ask for, as cases that can be timed.

A case names a mesh (square, L-shape or Kuhn cube, N vertices to a side), a
coefficient, a precision form of the solver and one call of the public API:

  grad      reduced_cost(u).backward(): state solve forward, adjoint solve backward
  hessian   Problem.hessian_apply of one control or of a block of them
  precond   Problem.precond_apply (the multilevel Hessian preconditioner) of one residual
  solve     Problem.solve: the outer CG on a problem that is set up
  block     Problem.solve_block: several desired states of one problem together
  step      Problem(...), amg_setup and solve: what one new mesh costs
  batch     Batch.solve: several problems with several desired states each
  inverse   dense_spd_inverse: the exact coarsest solve on its own

Inputs are made on the GPU from the seed alone.  Inner solves run to 1e-12 and
outer ones to 1e-10, so that an output is settled well below the accuracy that
users of the default tolerances see; the refinement form (precision 1), whose
FP32 inner CG does not reach as far at high contrast, runs at the defaults.
"""
import math

import torch

from paper_2001_11533_gb300 import amgh
from paper_2001_11533_gb300.autograd import reduced_cost

F64 = torch.float64


def _apply_opts(case):
    tol = 1e-10 if case["precision"] == 1 else 1e-12
    return dict(inner_tol=tol, mass_tol=tol, precond_tol=tol)


def _solve_opts(case):
    tol, inner = (1e-8, 1e-10) if case["precision"] == 1 else (1e-10, 1e-12)
    return dict(tol=tol, inner_tol=inner, mass_tol=1e-8, precond_tol=1e-8, level_fallback=1)


def listed():
    return [
        # the smallest problem of the tests, in the default FP64 form: one cost
        # and gradient of an optimiser's step, all launches and latency
        dict(name="grad_square33_fp64", op="grad", mesh="square", N=33, kappa="one", beta=1e-2, precision=0,
             coarse_max=256),
        # the smallest mesh of the batch workload, solved alone in the mixed form
        dict(name="solve_square65_mixed", op="solve", mesh="square", N=65, kappa="one", beta=1e-2, precision=2,
             coarse_max=256),
        # one control-sized Hessian product of a user's own Krylov method, FP64,
        # high-contrast L-shape of a quarter of the benchmark's side
        dict(name="hessian_lshape257_fp64", op="hessian", mesh="lshape", N=257, kappa="checker", beta=1e-4,
             precision=0, coarse_max=256, cols=1),
        # the refinement form on an L-shape of half the benchmark's side
        dict(name="hessian_lshape513_refine", op="hessian", mesh="lshape", N=513, kappa="checker", beta=1e-4,
             precision=1, coarse_max=256, cols=1),
        # the preconditioner alone, for a user's own outer iteration: all levels,
        # mass solves and small coarse solves
        dict(name="precond_square201_mixed", op="precond", mesh="square", N=201, kappa="one", beta=1e-2,
             precision=2, coarse_max=256),
        # eight desired states of one problem together (the batching pattern)
        dict(name="block8_square257_mixed", op="block", mesh="square", N=257, kappa="one", beta=1e-2, precision=2,
             coarse_max=1000, cols=8),
        # a small mesh from assembly to solution in the default form: setup counts
        dict(name="step_square129_fp64", op="step", mesh="square", N=129, kappa="one", beta=1e-2, precision=0,
             coarse_max=256),
        # the benchmark: 1025^2 L-shape from assembly to solution as it runs there
        dict(name="step_lshape1025_mixed", op="step", mesh="lshape", N=1025, kappa="checker", beta=1e-4, precision=2,
             coarse_max=1000, persistent=1),
        # cost and gradient on the random-field cube of the autograd tests, 3D rows
        dict(name="grad_cube65_mixed", op="grad", mesh="cube", N=65, kappa="grf", beta=1e-2, precision=2,
             coarse_max=256),
        # the largest: a Hessian product on the 129^3 cube (2 million states)
        dict(name="hessian_cube129_mixed", op="hessian", mesh="cube", N=129, kappa="grf", beta=1e-2, precision=2,
             coarse_max=256, cols=1),
        # uneven problems with several desired states each, run side by side
        dict(name="batch_squares_mixed", op="batch", mesh="square", N=129, kappa="one", beta=1e-2, precision=2,
             coarse_max=1000, cols=4, problems=4),
        # the dense coarsest inverse at the size that the benchmark's hierarchy ends with
        dict(name="inverse_847_fp64", op="inverse", N=847, precision=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choices(["grad", "hessian", "precond", "solve", "block", "step", "batch", "inverse"],
                     [3, 4, 2, 3, 2, 3, 1, 1])[0]
    if op == "inverse":
        return dict(op=op, N=_log_int(rng, 17, 1500), precision=0)
    mesh = rng.choice(["square", "lshape", "cube"])
    if op == "batch":
        mesh = "square"
    # sides: 2D 17 .. 513, 3D 9 .. 65 (a whole solve costs tens of applies)
    whole = op in ("solve", "block", "step", "batch")
    top2, top3 = (321, 41) if whole else (641, 97)
    if mesh == "cube":
        N = _log_int(rng, 9, top3)
    else:
        N = _log_int(rng, 17, 161 if op == "batch" else top2)
        if mesh == "lshape":
            N |= 1  # the re-entrant corner is a grid vertex
    kappa = {"square": "one", "lshape": "checker", "cube": rng.choice(["grf", "ball"])}[mesh]
    case = dict(op=op, mesh=mesh, N=N, kappa=kappa, beta=10.0 ** rng.uniform(-2.0, -0.5),
                precision=rng.choice([0, 0, 1, 2, 2, 2]), coarse_max=rng.choice([64, 256, 1000]))
    if op == "hessian":
        case["cols"] = rng.choice([1, 1, 2, 3, 5, 8])
    elif op == "block":
        case["cols"] = rng.choice([2, 3, 4, 7, 8])
    elif op == "batch":
        case["cols"] = rng.choice([1, 2, 3, 5])
        case["problems"] = rng.choice([1, 2, 3, 5])
    return case


# ------------------------------------------------------------------ inputs
def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + stream)
    return g


def _uniform(shape, lo, hi, gen):
    return torch.rand(shape, dtype=F64, device="cuda", generator=gen) * (hi - lo) + lo


def _square(N):
    """Vertices i + N j on [0, 1]^2, each square split along (i, j)-(i+1, j+1)."""
    v = torch.arange(N * N, device="cuda")
    coords = torch.stack([v % N, v // N], 1).to(F64) / (N - 1)
    c = torch.arange(N - 1, device="cuda")
    v00 = (c[None, :] + N * c[:, None]).reshape(-1)
    lower = torch.stack([v00, v00 + 1, v00 + N + 1], 1)
    upper = torch.stack([v00, v00 + N + 1, v00 + N], 1)
    elems = torch.stack([lower, upper], 1).reshape(-1, 3)
    i, j = v % N, v // N
    dirichlet = (i == 0) | (i == N - 1) | (j == 0) | (j == N - 1)
    return coords, elems, dirichlet


def _lshape(N):
    """The square without its upper right quarter (N odd)."""
    coords, elems, dirichlet = _square(N)
    mid = (N - 1) // 2
    v = torch.arange(N * N, device="cuda")
    i, j = v % N, v // N
    keep = ~((i > mid) & (j > mid))
    dirichlet = dirichlet | ((i == mid) & (j >= mid)) | ((j == mid) & (i >= mid))
    new = torch.cumsum(keep.to(torch.int64), 0) - 1
    return coords[keep], new[elems[keep[elems].all(1)]], dirichlet[keep]


def _cube(N):
    """Vertices i + N j + N^2 k on [0, 1]^3, six Kuhn tetrahedra per cell."""
    v = torch.arange(N ** 3, device="cuda")
    ijk = torch.stack([v % N, (v // N) % N, v // (N * N)], 1)
    c = torch.arange(N - 1, device="cuda")
    base = (c[None, None, :] + N * c[None, :, None] + N * N * c[:, None, None]).reshape(-1)
    step = (1, N, N * N)
    tets = []
    for a, b in ((0, 1), (0, 2), (1, 0), (1, 2), (2, 0), (2, 1)):
        tets.append(torch.stack([base, base + step[a], base + step[a] + step[b], base + 1 + N + N * N], 1))
    elems = torch.stack(tets, 1).reshape(-1, 4)
    return ijk.to(F64) / (N - 1), elems, ((ijk == 0) | (ijk == N - 1)).any(1)


def _kappa(kind, coords, elems, gen):
    if kind == "one":
        return torch.ones(elems.shape[0], dtype=F64, device="cuda")
    mid = coords[elems[:, 0]].clone()
    for k in range(1, elems.shape[1]):
        mid += coords[elems[:, k]]
    mid /= elems.shape[1]
    if kind == "checker":  # 1 or 1e4 on an 8 x 8 checkerboard
        cells = torch.rand(64, device="cuda", generator=gen) < 0.5
        at = (mid * 8).long().clamp(max=7)
        high = cells[at[:, 0] + 8 * at[:, 1]]
        return torch.where(high, 1e4, 1.0).to(F64)
    if kind == "ball":  # low coefficient in a ball that the mesh does not follow
        centre = _uniform((1, mid.shape[1]), 0.4, 0.6, gen)
        inside = ((mid - centre) ** 2).sum(1) <= 0.25 ** 2
        return torch.where(inside, 0.1, 1.0).to(F64)
    # exp of a Gaussian random field of correlation length 0.1, by random Fourier features
    F = 64
    omega = torch.randn((F, mid.shape[1]), dtype=F64, device="cuda", generator=gen) / 0.1
    phase = _uniform((F,), 0.0, 2.0 * math.pi, gen)
    field = torch.zeros(mid.shape[0], dtype=F64, device="cuda")
    for f in range(F):
        arg = mid[:, 0] * omega[f, 0] + phase[f]
        for d in range(1, mid.shape[1]):
            arg += mid[:, d] * omega[f, d]
        field += torch.cos(arg)
    return torch.exp(math.sqrt(2.0 / F) * field)


def _bumps(coords, cols, gen):
    """Desired states: sums of 8 Gaussian bumps of width 0.1, one row each."""
    out = torch.zeros((cols, coords.shape[0]), dtype=F64, device="cuda")
    for c in range(cols):
        centres = _uniform((8, coords.shape[1]), 0.0, 1.0, gen)
        amps = _uniform((8,), -1.0, 1.0, gen)
        for k in range(8):
            out[c] += amps[k] * torch.exp(-((coords - centres[k]) ** 2).sum(1) / 0.02)
    return out


def _inputs(case, seed):
    """Mesh, coefficient and desired states of one problem, as tensors on the GPU."""
    mesh, N = case["mesh"], case["N"]
    coords, elems, dirichlet = {"square": _square, "lshape": _lshape, "cube": _cube}[mesh](N)
    gen = _gen(seed, 1)
    if mesh != "cube":  # interior vertices moved by up to a fifth of the mesh width
        move = _uniform(coords.shape, -0.2 / (N - 1), 0.2 / (N - 1), gen)
        coords = coords + torch.where(dirichlet[:, None], 0.0, move)
    kappa = _kappa(case["kappa"], coords, elems, gen)
    yd = _bumps(coords, case.get("cols", 1), gen)
    return dict(dim=coords.shape[1], coords=coords.contiguous(), elems=elems.to(torch.int32).contiguous(),
                dirichlet=dirichlet.to(torch.uint8), kappa=kappa, beta=case["beta"], yd=yd)


def _problem(w):
    return amgh.Problem(w["dim"], w["coords"], w["elems"], w["dirichlet"], w["kappa"], w["beta"], w["yd"][0],
                        on_device=True)


def _setup_opts(case):
    return dict(precision=case["precision"], coarse_max=case["coarse_max"], coarse_solve=2,
                persistent_cg=case.get("persistent", 0))


def _controls(w, cols, seed):
    """Control-sized vectors with smooth and rough parts, one row each."""
    gen = _gen(seed, 2)
    n = w["coords"].shape[0]
    return _bumps(w["coords"], cols, gen) + 0.1 * torch.randn((cols, n), dtype=F64, device="cuda", generator=gen)


def _spd(N, seed):
    """A symmetric positive definite matrix with eigenvalues in about [1, 100]."""
    gen = _gen(seed, 3)
    B = torch.randn((N, N), dtype=F64, device="cuda", generator=gen)
    d = torch.exp(_uniform((N,), 0.0, math.log(30.0), gen))
    return B @ B.T / N + torch.diag(d) + torch.eye(N, dtype=F64, device="cuda")


def _batch_inputs(case, seed):
    """Problems of uneven size: sides N, N/2, N/4, ... (at least 9), then again."""
    sides = [max(9, case["N"] >> k) | 1 for k in range(3)]
    return [_inputs(dict(case, N=sides[i % 3], beta=case["beta"] * (1 + i)), 101 * seed + i)
            for i in range(case["problems"])]


def prepare(case, seed):
    op = case["op"]
    state = dict(op=op, case=case)
    if op == "inverse":
        state["a"] = _spd(case["N"], seed)
        return state
    if op == "batch":
        ws = _batch_inputs(case, seed)
        state["yds"] = [w["yd"] for w in ws]
        torch.cuda.synchronize()
        state["batch"] = amgh.Batch([_problem(w) for w in ws]).setup(**_setup_opts(case))
        return state
    w = _inputs(case, seed)
    torch.cuda.synchronize()
    if op == "step":
        state["w"] = w
        return state
    p = _problem(w).amg_setup(**_setup_opts(case))
    p.set_solve_opts(**_apply_opts(case))
    state["p"] = p
    if op == "block":
        state["yd"] = w["yd"]
    elif op in ("grad", "hessian", "precond"):
        u = _controls(w, case.get("cols", 1), seed)
        state["u"] = u if case.get("cols", 1) > 1 else u[0].contiguous()
    return state


def run(state):
    op = state["op"]
    if op == "grad":
        u = state["u"].detach().requires_grad_(True)
        J = reduced_cost(u, state["p"])
        J.backward()
        return [J, u.grad]
    if op == "hessian":
        return state["p"].hessian_apply(state["u"])
    if op == "precond":
        return state["p"].precond_apply(state["u"])
    if op == "solve":
        u, y, _ = state["p"].solve(**_solve_opts(state["case"]))
        return [u, y]
    if op == "block":
        return state["p"].solve_block(state["yd"], **_solve_opts(state["case"]))[0]
    if op == "step":
        p = _problem(state["w"]).amg_setup(**_setup_opts(state["case"]))
        u, y, _ = p.solve(**_solve_opts(state["case"]))
        p.close()
        return [u, y]
    if op == "batch":
        return state["batch"].solve(state["yds"], **_solve_opts(state["case"]))[0]
    inv = torch.empty_like(state["a"])
    status, info = amgh.dense_spd_inverse(state["a"], inv)
    return [inv, status, info]


# ------------------------------------------------------------------ compulsory work
def _counts(case):
    """Vertices, elements and stored entries of one assembled matrix."""
    N = case["N"]
    if case["mesh"] == "cube":
        return N ** 3, 6 * (N - 1) ** 3, 15 * N ** 3
    f = 0.75 if case["mesh"] == "lshape" else 1.0
    return int(f * N * N), int(f * 2 * (N - 1) ** 2), int(f * 7 * N * N)


def work(case):
    """The inputs read once, the outputs written once, and one product with each
    operator of the path per column: the solves' iterations are the method's own."""
    op, cols = case["op"], case.get("cols", 1)
    if op == "inverse":
        n = case["N"]
        return {"bytes": 16.0 * n * n, "flops": 2.0 * n ** 3}
    if op == "batch":
        sides = [max(9, case["N"] >> k) | 1 for k in range(3)]
        parts = [work(dict(case, op="block", N=sides[i % 3])) for i in range(case["problems"])]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n, ne, nnz = _counts(case)
    dim = 3 if case["mesh"] == "cube" else 2
    operators = 12.0 * 3 * nnz  # stiffness, mass and cross mass: 8-byte values, 4-byte columns
    b, f = operators + 8.0 * n * 3 * cols, 2.0 * 7 * nnz * cols
    if op in ("solve", "block", "step"):
        f *= 4
    if op == "step":
        b += 8.0 * dim * n + ne * (4.0 * (dim + 1) + 8.0)
        f += ne * (dim + 1) ** 2 * 10.0
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ values in 64 bits
class _Dense64:
    """The discrete problem in plain torch FP64: P1 stiffness and mass in CSR over
    all vertices, Dirichlet rows masked."""

    def __init__(self, w):
        X = w["coords"][w["elems"].long()]
        d = w["dim"]
        E = X[:, 1:, :] - X[:, :1, :]
        # gradients of the barycentric coordinates 1..d: the columns of E^-1
        if d == 2:
            det = E[:, 0, 0] * E[:, 1, 1] - E[:, 0, 1] * E[:, 1, 0]
            G = torch.stack([torch.stack([E[:, 1, 1], -E[:, 1, 0]], 1),
                             torch.stack([-E[:, 0, 1], E[:, 0, 0]], 1)], 2)
        else:
            c = [torch.linalg.cross(E[:, (k + 1) % 3], E[:, (k + 2) % 3]) for k in range(3)]
            det = (E[:, 0] * c[0]).sum(1)
            G = torch.stack(c, 2)
        G = G / det[:, None, None]
        vol = det.abs() / math.factorial(d)
        G = torch.cat([-G.sum(2, keepdim=True), G], 2)
        Ke = (w["kappa"] * vol)[:, None, None] * (G.transpose(1, 2) @ G)
        Me = (torch.ones((d + 1, d + 1), dtype=F64, device="cuda") + torch.eye(d + 1, dtype=F64, device="cuda"))
        Me = vol[:, None, None] / ((d + 1) * (d + 2)) * Me
        n, e = w["coords"].shape[0], w["elems"].long()
        rows = e[:, :, None].expand(-1, d + 1, d + 1).reshape(-1)
        cols = e[:, None, :].expand(-1, d + 1, d + 1).reshape(-1)

        def csr(vals):
            A = torch.sparse_coo_tensor(torch.stack([rows, cols]), vals.reshape(-1), (n, n))
            return A.coalesce().to_sparse_csr()

        self.K, self.M = csr(Ke), csr(Me)
        self.free = (w["dirichlet"] == 0).to(F64)[:, None]
        diag = torch.zeros(n, dtype=F64, device="cuda")
        diag.index_add_(0, e.reshape(-1), torch.diagonal(Ke, dim1=1, dim2=2).reshape(-1))
        self.dinv = torch.where(self.free > 0, 1.0 / diag[:, None], 0.0)
        self.beta = w["beta"]

    @staticmethod
    def cg(mul, dinv, b, tol, most):
        """Preconditioned CG on the columns of b, each with its own scalars."""
        x = torch.zeros_like(b)
        r = b.clone()
        z = dinv * r
        p = z.clone()
        rz = (r * z).sum(0)
        stop = tol * tol * (r * r).sum(0)
        for k in range(most):
            q = mul(p)
            pq = (p * q).sum(0)
            a = torch.where(pq > 0, rz / pq.clamp(min=1e-300), 0.0)
            x += a * p
            r -= a * q
            z = dinv * r
            new = (r * z).sum(0)
            p = z + torch.where(rz > 0, new / rz.clamp(min=1e-300), 0.0) * p
            rz = new
            if k % 25 == 24 and bool(((r * r).sum(0) <= stop).all()):
                break
        return x

    def state(self, f):
        """A^-1 f on the free vertices, with one step of refinement."""
        mul = lambda v: self.free * (self.K @ v)  # noqa: E731
        y = self.cg(mul, self.dinv, self.free * f, 1e-13, 20000)
        return y + self.cg(mul, self.dinv, self.free * f - mul(y), 1e-6, 20000)

    def hessian(self, u):
        y = self.state(self.M @ u)
        return self.M @ self.state(self.M @ y) + self.beta * (self.M @ u)

    def rhs(self, yd):
        return self.M @ self.state(self.M @ (self.free * yd))

    def control(self, yd):
        """The optimal control: CG on H u = b, to well below the tolerance of a solve."""
        lump = self.M @ torch.ones_like(self.free)
        return self.cg(self.hessian, 1.0 / lump, self.rhs(yd), 1e-13, 100)


def _exact_control(w):
    D = _Dense64(w)
    u = D.control(w["yd"].T.contiguous())
    y = D.state(D.M @ u)
    return u, y, D.free[:, 0] > 0


def exact(case, seed):
    """Plain torch in FP64.  None for the preconditioner, whose value depends on the
    hierarchy, and for whole solves on meshes where plain CG takes too long."""
    op = case["op"]
    if op == "inverse":
        return [torch.linalg.inv(_spd(case["N"], seed)), None, None]
    if op == "precond":
        return None
    most = 30000 if case["kappa"] == "one" else 5000
    if op == "batch":
        ws = _batch_inputs(case, seed)
        if sum(w["coords"].shape[0] for w in ws) > most:
            return None
        return [_exact_control(w)[0].T.contiguous() for w in ws]
    n = _counts(case)[0]
    if op in ("solve", "block", "step"):
        if n * (1 if case["mesh"] != "cube" else 0.2) > most:
            return None
        w = _inputs(case, seed)
        u, y, free = _exact_control(w)
        if op == "block":
            return u.T.contiguous()
        return [u[:, 0].contiguous(), y[free, 0].contiguous()]
    w = _inputs(case, seed)
    D = _Dense64(w)
    u = _controls(w, case.get("cols", 1), seed).T.contiguous()
    if op == "hessian":
        hu = D.hessian(u).T.contiguous()
        return hu if case.get("cols", 1) > 1 else hu[0].contiguous()
    yd = w["yd"].T.contiguous()
    y = D.state(D.M @ u)
    e = y - D.free * yd
    J = 0.5 * (e * (D.M @ e)).sum() + 0.5 * w["beta"] * (u * (D.M @ u)).sum()
    g = D.M @ D.state(D.M @ e) + w["beta"] * (D.M @ u)
    return [J, g[:, 0].contiguous()]
