"""What a user of this package has it do, as cases that can be timed and compared.

The package solves the Newton systems J(psi) x = b of the extreme type-II
Ginzburg-Landau problem (Schloemer & Vanroose, arXiv:1204.5125).  A program makes
a mesh, sets up the multigrid preconditioner for a state psi, and then applies
operators, solves, takes Newton steps, runs batches, or trains and evaluates the
learned initial guess.  Each case below is one such call through the public entry
points; meshes, preconditioners, batches and network handles are made beforehand
(`prepare`), as a program that keeps them would, except in the Newton step, whose
call sets up its own preconditioner.

A case is a dict:
  op       jacobian | residual | precond | solve | newton | batch | predict | grad
  mesh     square | cube (the paper's square and cube of circumradius 5 as lattices) |
           hex (a general simplicial mesh of that square: a jittered triangular lattice)
  N        nodes per side
  precision  fp64 | mixed (FP32 V-cycle inside FP64 MINRES)
  mu       field strength (the field along z on squares, along (1,1,1) on cubes)
  coarse   size at which the hierarchy stops coarsening
  count    systems of a batch (N is then the largest side, the others are spread
           below it)
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

import paper_1204_5125_gb300 as gl

PREC = {"fp64": gl.GL_FP64, "mixed": gl.GL_MIXED_PRECOND}
DEV = "cuda"
# sides of the square and the cube of circumradius 5
EDGE = {"square": 10 / math.sqrt(2.0), "hex": 10 / math.sqrt(2.0), "cube": 10 / math.sqrt(3.0)}


def listed():
    return [
        # one operator apply on the smallest mesh in use: a user's own Krylov or
        # eigenvalue loop on a small problem, bound by the call itself
        dict(name="jacobian_square64", op="jacobian", mesh="square", N=64, mu=1.0),
        # the same on the benchmark's cube: the operator at streaming size
        dict(name="jacobian_cube128", op="jacobian", mesh="cube", N=128, mu=1.0),
        # the nonlinear residual that every Newton iteration starts with, odd side
        dict(name="residual_square1023", op="residual", mesh="square", N=1023, mu=2.0),
        # one preconditioner application for a user's own Krylov method: an odd
        # cube, where the finest level works from the stored matrix, in FP64
        dict(name="precond_cube97", op="precond", mesh="cube", N=97, mu=1.0, coarse=4096),
        # the paper's plain FP64 solve on a small square (latency)
        dict(name="solve_square64", op="solve", mesh="square", N=64, mu=1.0, precision="fp64", coarse=512),
        # a solve on a large square at a field strength where many vortices form,
        # mixed precision: three levels, many iterations
        dict(name="solve_square1024", op="solve", mesh="square", N=1024, mu=2.0, precision="mixed", coarse=512),
        # the headline workload: the 128^3 cube, mixed precision
        dict(name="solve_cube128", op="solve", mesh="cube", N=128, mu=1.0, precision="mixed", coarse=4096),
        # FP64 solve on a general triangulation (the paper's own kind of mesh):
        # stored matrix, many-coloured finest level
        dict(name="solve_hex150", op="solve", mesh="hex", N=150, mu=1.0, precision="fp64", coarse=512),
        # a whole Newton step with its preconditioner setup: the inner loop of a
        # continuation, on the benchmark's cube
        dict(name="newton_cube128", op="newton", mesh="cube", N=128, mu=1.0, precision="mixed", coarse=4096),
        # independent systems of uneven sizes in one launch (parameter sweeps)
        dict(name="batch12_square320", op="batch", mesh="square", N=320, mu=2.0, precision="mixed", coarse=512,
             count=12),
        # inference of the learned initial guess on the benchmark's cube
        dict(name="predict_cube128", op="predict", mesh="cube", N=128, mu=1.0),
        # loss and gradient of one training sample, odd cube (a ragged last tile)
        dict(name="grad_cube63", op="grad", mesh="cube", N=63, mu=1.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["jacobian", "jacobian", "residual", "precond", "solve", "solve", "solve", "newton", "batch",
                     "predict", "grad"])
    mu = round(rng.uniform(0.5, 2.0), 3)
    if op == "batch":
        return dict(op=op, mesh="square", N=_log_int(rng, 48, 320), mu=mu, precision=rng.choice(["fp64", "mixed"]),
                    coarse=512, count=rng.randint(3, 12))
    mesh = rng.choice(["square", "cube", "cube", "hex"])
    if op in ("predict", "grad"):
        mesh = rng.choice(["square", "cube"])
    lo, hi = {"square": (32, 1023), "cube": (16, 128), "hex": (32, 400)}[mesh]
    if op in ("newton", "grad"):
        hi = {"square": 512, "cube": 96, "hex": 256}[mesh]
    case = dict(op=op, mesh=mesh, N=_log_int(rng, lo, hi), mu=mu)
    if op in ("precond", "solve", "newton"):
        case["coarse"] = rng.choice([512, 4096]) if mesh == "cube" else 512
    if op in ("solve", "newton"):
        case["precision"] = "fp64" if mesh == "hex" else rng.choice(["fp64", "mixed"])
    return case


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _normal(n, g):
    """Complex normal, variance 1."""
    return torch.view_as_complex(torch.randn(n, 2, dtype=torch.float64, device=DEV, generator=g) / math.sqrt(2.0))


def _near_one(n, g):
    """1 + 0.1 (uniform in the unit disk): a state on the way to a solution."""
    u = torch.rand(2, n, dtype=torch.float64, device=DEV, generator=g)
    return 1.0 + 0.1 * torch.polar(torch.sqrt(u[0]), 2.0 * math.pi * u[1])


def _nodes(case):
    return case["N"] ** (3 if case["mesh"] == "cube" else 2)


def _bhat(case):
    return (3.0 ** -0.5,) * 3 if case["mesh"] == "cube" else (0.0, 0.0, 1.0)


def _hex_mesh(N, seed):
    """N x N nodes of an equilateral triangular lattice, every node moved by up to a
    tenth of the spacing, and its triangles (which stay Delaunay)."""
    L = EDGE["hex"]
    h = L / (N - 1)
    j, i = np.divmod(np.arange(N * N), N)
    x = np.stack([(i + 0.5 * (j % 2)) * h - 0.5 * L, (j * h - 0.5 * L) * math.sqrt(0.75), np.zeros(N * N)], axis=1)
    x[:, :2] += np.random.default_rng(seed).uniform(-0.07 * h, 0.07 * h, (N * N, 2))
    a = (np.arange(N - 1)[:, None] * N + np.arange(N - 1)[None, :]).ravel()
    odd = (a // N) % 2 == 1
    lower = np.where(odd[:, None], np.stack([a, a + 1, a + N + 1], 1), np.stack([a, a + 1, a + N], 1))
    upper = np.where(odd[:, None], np.stack([a, a + N + 1, a + N], 1), np.stack([a + 1, a + N + 1, a + N], 1))
    return x, np.concatenate([lower, upper]).astype(np.int32)


def _network(seed):
    """Parameters of the learned guess as training starts from them: He-normal layers
    and a small head."""
    r = np.random.default_rng(seed)
    layers = r.standard_normal(4 * 64 * 128) * math.sqrt(2.0 / 128)
    return np.concatenate([layers, r.standard_normal(2 * 64) * (0.1 / 8.0)]).astype(np.float32)


def _batch_sides(case):
    k = case["count"]
    return [max(24, int(case["N"] * (0.3 + 0.7 * (i + 1) / k))) for i in range(k)]


class _State:
    """Inputs and the handles a program keeps; the handles go with it."""

    def __init__(self):
        self.meshes, self.prec, self.batch, self.ws = [], None, None, None

    def __del__(self):
        if self.prec is not None:
            gl.gl_precond_destroy(self.prec)
        if self.batch is not None:
            gl.gl_batch_destroy(self.batch)
        if self.ws is not None:
            gl.gl_warmstart_destroy(self.ws)
        for m in self.meshes:
            gl.gl_mesh_destroy(m)


def prepare(case, seed):
    s, g, op = _State(), _gen(seed), case["op"]
    s.op = op
    s.options = gl.options(precision=PREC[case.get("precision", "fp64")], max_coarse=case.get("coarse", 512))
    if op == "batch":
        sides = _batch_sides(case)
        s.meshes = [gl.gl_mesh_create(2, k, case["mu"] * (0.5 + 0.5 * (i + 1) / len(sides)), edge=EDGE["square"])
                    for i, k in enumerate(sides)]
        psi = [_near_one(k * k, g) for k in sides]
        s.b = [_normal(k * k, g) for k in sides]
        s.batch = gl.gl_batch_create(s.meshes, psi, s.options)
        s.x = [torch.zeros_like(b) for b in s.b]
        return s
    n = _nodes(case)
    if case["mesh"] == "hex":
        x, simplices = _hex_mesh(case["N"], seed)
        s.meshes = [gl.gl_mesh_create_simplicial(2, x, simplices, case["mu"])]
    else:
        s.meshes = [gl.gl_mesh_create(3 if case["mesh"] == "cube" else 2, case["N"], case["mu"], _bhat(case),
                                      edge=EDGE[case["mesh"]])]
    s.mesh = s.meshes[0]
    s.psi = _near_one(n, g)
    if op not in ("residual", "newton"):
        s.b = _normal(n, g)
    if op in ("precond", "solve"):
        s.prec = gl.gl_precond_setup(s.mesh, s.psi, s.options)
    if op in ("predict", "grad"):
        s.ws = gl.gl_warmstart_create(_network(seed))
    return s


def run(s):
    if s.op == "jacobian":
        y = torch.empty_like(s.b)
        gl.gl_jacobian_apply(s.mesh, s.psi, s.b, y)
        return y
    if s.op == "residual":
        r = torch.empty_like(s.psi)
        gl.gl_residual(s.mesh, s.psi, r)
        return r
    if s.op == "precond":
        z = torch.empty_like(s.b)
        gl.gl_precond_apply(s.prec, s.b, z)
        return z
    if s.op == "solve":
        x = torch.zeros_like(s.b)
        gl.gl_jacobian_solve(s.mesh, s.psi, s.prec, s.b, x, s.options)
        return x
    if s.op == "newton":
        psi = s.psi.clone()
        _, _, norm = gl.gl_newton_step(s.mesh, psi, s.options)
        return {"psi": psi, "norm": norm}
    if s.op == "batch":
        for x in s.x:
            x.zero_()
        gl.gl_batch_run(s.batch, s.b, s.x)
        return s.x
    if s.op == "predict":
        x0 = torch.empty_like(s.b)
        gl.gl_warmstart_predict(s.ws, s.mesh, s.psi, s.b, x0)
        return x0
    loss, grad = gl.gl_warmstart_grad(s.ws, s.mesh, s.psi, s.b)
    return {"loss": loss, "grad": grad}


# ---------------------------------------------------------------- work
ITERATIONS = 18  # MINRES iterations that a solve to 1e-10 takes at the least over these ranges


def _vcycle_work(n, entries, real):
    """(bytes, flops) of one V-cycle's finest level, a third of it again below: two
    symmetric Gauss-Seidel steps and a residual (four sweeps' worth of flops; the
    right-hand side and diagonal read and the vector written), `real` bytes a real."""
    return 4 / 3 * n * 5 * real, 4 / 3 * (4 * 8 * entries + 40 * n)


def work(case):
    """Bytes and flops of one pass.  The bytes count each vector of a step once in and
    once out; stored matrix entries are not counted on lattices, whose few distinct
    edge values fit in cache, and are counted (value and column) on general meshes."""
    ns = [k * k for k in _batch_sides(case)] if case["op"] == "batch" else [_nodes(case)]
    deg = {"square": 4, "cube": 6, "hex": 6}[case["mesh"]]
    op, total_b, total_f = case["op"], 0.0, 0.0
    for n in ns:
        stored = deg * n * 20 if case["mesh"] == "hex" else 0
        jac = (48.0 * n + stored, (8 * deg + 20) * n)
        real = 4 if case.get("precision") == "mixed" else 8
        vcb, vcf = _vcycle_work(n, deg * n, real)
        vcb += stored
        if op == "jacobian":
            b, f = jac
        elif op == "residual":
            b, f = 32.0 * n + stored, (8 * deg + 8) * n
        elif op == "precond":
            b, f = vcb, vcf
        elif op in ("solve", "newton", "batch"):
            # per iteration one Jacobian, one V-cycle and the three recurrences
            b = ITERATIONS * (jac[0] + vcb + 14 * 16.0 * n) + 48.0 * n
            f = ITERATIONS * (jac[1] + vcf + 40.0 * n)
        else:
            # four layers of 64 channels (BF16 activations in and out, one 64 x 128
            # product a node), twice as much again backward
            layers = 1 if op == "predict" else 3
            b = layers * 4 * 2 * 128.0 * n + 64.0 * n
            f = layers * 4 * 2.0 * 64 * 128 * n
        total_b += b
        total_f += f
    return {"bytes": total_b, "flops": total_f}


# ---------------------------------------------------------------- 64-bit results
class _Lattice:
    """K psi of the square or cube lattice from Eq. (10): coefficients of the Kuhn
    split, phases (mu/2) h B . (x_j x e), control volumes h^d 2^-b."""

    def __init__(self, case):
        self.d, self.N = (3 if case["mesh"] == "cube" else 2), case["N"]
        d, N, L = self.d, self.N, EDGE[case["mesh"]]
        h = L / (N - 1)
        f64 = dict(dtype=torch.float64, device=DEV)
        self.shape = (N,) * d  # axis order (z, y, x): x fastest
        pos = torch.arange(N, **f64) * h - 0.5 * L
        grid = torch.meshgrid(*([pos] * d), indexing="ij")[::-1]  # x, y[, z]
        X = [grid[e] if e < d else torch.zeros(self.shape, **f64) for e in range(3)]
        B = torch.tensor(_bhat(case), **f64)
        side = torch.full((N,), 0.0, **f64)
        side[0] = side[-1] = 1.0
        on = [side.reshape([N if a == d - 1 - e else 1 for a in range(d)]) for e in range(d)]
        self.vol = h ** d * torch.pow(2.0, -sum(o.expand(self.shape) for o in on))
        self.edges = []  # per axis: -alpha exp(-i theta) of the edge to the next node
        self.diag = torch.zeros(self.shape, **f64)
        for e in range(d):
            alpha = torch.zeros(self.shape, **f64)
            perp = [a for a in range(d) if a != e]
            # the cells around an edge: it is corner c of the cell at its own position - c
            for c in itertools.product((0, 1), repeat=d - 1):
                inside = torch.ones(self.shape, dtype=torch.bool, device=DEV)
                for a, ca in zip(perp, c):
                    k = torch.arange(N, device=DEV).reshape([N if q == d - 1 - a else 1 for q in range(d)])
                    inside = inside & ((k - ca >= 0) & (k - ca <= N - 2))
                share = 0.5 if d == 2 else (h / 3 if c in ((0, 0), (1, 1)) else h / 6)
                alpha += share * inside
            cross = {0: X[2] * B[1] - X[1] * B[2], 1: X[0] * B[2] - X[2] * B[0], 2: X[1] * B[0] - X[0] * B[1]}[e]
            theta = 0.5 * case["mu"] * h * cross  # B . (x x e)
            dim = d - 1 - e
            w = torch.polar(alpha, -theta).narrow(dim, 0, N - 1)
            self.edges.append((dim, w))
            a = alpha.narrow(dim, 0, N - 1)
            self.diag.narrow(dim, 0, N - 1).add_(a)
            self.diag.narrow(dim, 1, N - 1).add_(a)

    def off(self, u):
        """The off-diagonal part of K-hat u; u may carry trailing dimensions."""
        N, more = self.N, (1,) * (u.dim() - self.d)
        out = torch.zeros_like(u)
        for dim, w in self.edges:
            w = w.reshape(w.shape + more)
            out.narrow(dim, 0, N - 1).sub_(w * u.narrow(dim, 1, N - 1))
            out.narrow(dim, 1, N - 1).sub_(w.conj() * u.narrow(dim, 0, N - 1))
        return out

    def K(self, u):
        return (self.off(u) + self.diag * u) / self.vol

    def jacobian(self, psi, phi):
        return self.K(phi) + (2.0 * psi.abs() ** 2 - 1.0) * phi + psi * psi * phi.conj()

    def residual(self, psi):
        return self.K(psi) - psi * (1.0 - psi.abs() ** 2)

    def solve(self, psi, b):
        """J(psi) x = b as the dense real system of twice the size."""
        n = psi.numel()
        A = torch.empty(2 * n, 2 * n, dtype=torch.float64, device=DEV)
        for lo in range(0, 2 * n, 512):
            k = torch.arange(lo, min(lo + 512, 2 * n), device=DEV)
            unit = torch.zeros(n, len(k), dtype=torch.complex128, device=DEV)
            unit[k % n, torch.arange(len(k), device=DEV)] = torch.where(k < n, 1.0 + 0j, 1j).to(torch.complex128)
            u = unit.reshape(self.shape + (len(k),))
            p, one = psi.reshape(self.shape + (1,)), (1,)
            y = (self.off(u) + self.diag.reshape(self.shape + one) * u) / self.vol.reshape(self.shape + one)
            y = (y + (2.0 * p.abs() ** 2 - 1.0) * u + p * p * u.conj()).reshape(n, len(k))
            A[:n, k], A[n:, k] = y.real, y.imag
        x = torch.linalg.solve(A, torch.cat([b.real, b.imag]))
        return torch.complex(x[:n], x[n:])


def _network_guess(L, theta, psi, bhat):
    """x^ = y(psi, b^) / K_ii of the four-layer network, in FP64 (differentiable)."""
    Ws, U = theta[: 4 * 64 * 128].reshape(4, 64, 128), theta[4 * 64 * 128:].reshape(2, 64)
    n = psi.numel()
    h = torch.zeros(n, 64, dtype=torch.float64, device=DEV)
    h[:, 0], h[:, 1], h[:, 2], h[:, 3], h[:, 4] = bhat.real, bhat.imag, psi.real, psi.imag, psi.abs() ** 2
    h[:, 63] = 1.0
    for W in Ws:
        pairs = torch.view_as_complex(h.reshape(n, 32, 2)).reshape(L.shape + (32,))
        agg = -_Off.apply(L, pairs) / L.diag.reshape(L.shape + (1,))
        agg = torch.view_as_real(agg.reshape(n, 32)).reshape(n, 64)
        h = torch.relu(torch.cat([h, agg], dim=1) @ W.T)
        h = torch.cat([h[:, :63], torch.ones_like(h[:, :1])], dim=1)
    y = h @ U.T
    return torch.complex(y[:, 0], y[:, 1]) / (L.diag / L.vol).reshape(-1)


class _Off(torch.autograd.Function):
    @staticmethod
    def forward(ctx, L, u):
        ctx.L = L
        return L.off(u)

    @staticmethod
    def backward(ctx, g):
        return None, ctx.L.off(g)  # K-hat is Hermitian


class _Jac(torch.autograd.Function):
    @staticmethod
    def forward(ctx, L, psi, x):
        ctx.L, ctx.psi = L, psi
        return L.jacobian(psi, x)

    @staticmethod
    def backward(ctx, g):
        L = ctx.L  # D J is symmetric as a real operator
        return None, None, L.vol * L.jacobian(ctx.psi, g / L.vol)


def exact(case, seed):
    op, n = case["op"], _nodes(case)
    if case["mesh"] == "hex" or op in ("precond", "batch"):
        return None
    if op in ("solve", "newton") and n > 4096:
        return None
    L, g = _Lattice(case), _gen(seed)
    psi = _near_one(n, g).reshape(L.shape)
    if op == "residual":
        return L.residual(psi).reshape(-1)
    if op == "newton":
        r = L.residual(psi)
        return {"psi": psi.reshape(-1) + L.solve(psi, -r.reshape(-1)),
                "norm": float(torch.sqrt((L.vol * r.abs() ** 2).sum()))}
    b = _normal(n, g).reshape(L.shape)
    if op == "solve":
        return L.solve(psi, b.reshape(-1))
    if op == "jacobian":
        return L.jacobian(psi, b).reshape(-1)
    norm = torch.sqrt((L.vol * b.abs() ** 2).sum())
    theta = torch.from_numpy(_network(seed)).to(DEV).double().requires_grad_(op == "grad")
    bhat = b.reshape(-1) / norm
    x = _network_guess(L, theta, psi.reshape(-1), bhat)
    if op == "predict":
        return norm * x
    r = bhat.reshape(L.shape) - _Jac.apply(L, psi, x.reshape(L.shape))
    loss = (L.vol * (r.real ** 2 + r.imag ** 2)).sum()
    loss.backward()
    return {"loss": float(loss), "grad": theta.grad.cpu().numpy()}
