"""The performance cases of the bake-off library: the calls that its users make, with their sizes.

A user sets a problem up once (mesh, order, arithmetic), keeps the ``Operator`` or ``Batch`` and then
solves, applies the operator, or differentiates with respect to the coefficient, again and again.  Every
case here does one such call.  The sizes are those of the bake-off sweep (orders 1..15, about 1e4 to 2e7
degrees of freedom) and of the benchmark's configurations; the boxes of elements are not all cubes and
not all powers of two.

The mesh handed to the library (the deformed unit cube with its local-to-global map) and the reference
results of ``exact`` are computed in this file with numpy and torch alone.
"""
import math

import numpy as np
import torch

import paper_2004_06722_gb300 as ceedbp

AMP = 0.05  # deformation amplitude of the bake-off mesh


def listed():
    return [
        # one operator application on the 22k-DOF problem of the first configuration: launch latency
        dict(name="apply_bp5_n7_e64", op="apply", bp=5, order=7, ex=4, ey=4, ez=4, arith=0),
        # the first configuration: a whole solve to 1e-8 on the same mesh (many tiny launches)
        dict(name="solve_bp5_n7_e64_tol", op="solve", bp=5, order=7, ex=4, ey=4, ez=4, arith=0, tol=1e-8, iters=0),
        # the headline: 100 fixed CG iterations of BP5 at N = 7, native FP64 and FP32 pairs
        dict(name="solve_bp5_n7_large", op="solve", bp=5, order=7, ex=64, ey=32, ez=32, arith=0, tol=0.0, iters=100),
        dict(name="solve_bp5_n7_large_pairs", op="solve", bp=5, order=7, ex=64, ey=32, ez=32, arith=1, tol=0.0,
             iters=100),
        # Gauss quadrature stiffness, FP64 at the headline order, and pairs on a ragged mesh at a lower order
        dict(name="solve_bp3_n7", op="solve", bp=3, order=7, ex=25, ey=25, ez=25, arith=0, tol=0.0, iters=50),
        dict(name="solve_bp3_n5_pairs", op="solve", bp=3, order=5, ex=27, ey=25, ez=23, arith=1, tol=0.0, iters=50),
        # the mass problem at a low order, many elements
        dict(name="solve_bp1_n3", op="solve", bp=1, order=3, ex=41, ey=37, ez=29, arith=0, tol=0.0, iters=50),
        # BP5 at a high order, medium size
        dict(name="solve_bp5_n11", op="solve", bp=5, order=11, ex=17, ey=16, ez=15, arith=0, tol=0.0, iters=50),
        # unassembled element operator at an even order (the BK sweep)
        dict(name="bk5_n6", op="bk", bp=5, order=6, ex=21, ey=19, ez=17, arith=0),
        # vector Poisson by FP32 defect correction to 1e-10
        dict(name="mixed_bp6_n7", op="mixed", bp=6, order=7, ex=12, ey=12, ez=12, arith=0, precision="fp32"),
        # independent problems of uneven size and order, solved together to 1e-8
        dict(name="batch_fp64", op="batch", problems=32, kmin=2, kmax=12, arith=0),
        # forward solve, adjoint solve and coefficient gradient to 1e-10
        dict(name="adjoint_n7", op="adjoint", bp=5, order=7, ex=12, ey=12, ez=12, arith=0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _box(rng, order, lo, hi):
    """Elements in each direction of a box with about lo..hi degrees of freedom (E N^3)."""
    e = max(1.0, _log(rng, lo, hi) / order ** 3)
    k = e ** (1.0 / 3.0)
    ex = max(1, round(k * _log(rng, 0.75, 1.33)))
    ey = max(1, round(k * _log(rng, 0.75, 1.33)))
    return ex, ey, max(1, round(e / (ex * ey)))


def draw(rng):
    op = rng.choice(["solve"] * 6 + ["apply"] * 3 + ["bk"] * 2 + ["mixed", "batch", "adjoint"])
    if op == "batch":
        return dict(op=op, problems=rng.randint(8, 32), kmin=2, kmax=rng.randint(6, 12), arith=rng.randint(0, 1))
    if op == "mixed":
        order = rng.choice([3, 5, 6, 7, 8])
        ex, ey, ez = _box(rng, order, 2e4, 6e5)
        return dict(op=op, bp=rng.choice([5, 6]), order=order, ex=ex, ey=ey, ez=ez, arith=0,
                    precision=rng.choice(["fp32", "fp32", "bf16"]))
    if op == "adjoint":
        order = rng.choice([4, 5, 7, 9])
        ex, ey, ez = _box(rng, order, 2e4, 6e5)
        return dict(op=op, bp=5, order=order, ex=ex, ey=ey, ez=ez, arith=0)
    bp = rng.choice([1, 3, 3, 5, 5, 5, 6] if rng.random() < 0.9 else [2, 4])
    arith = 1 if bp not in (2, 4) and rng.random() < 0.35 else 0
    order = rng.choice([1, 2, 3, 3, 4, 5, 5, 6, 7, 7, 7, 8, 9, 9, 10, 11, 11, 12, 13, 14, 15, 15])
    top = 8e6 / (3 if bp in (2, 4, 6) else 1) / (2 if bp in (3, 4) else 1)
    if order < 3:
        top /= 8  # local nodes outnumber the degrees of freedom
    ex, ey, ez = _box(rng, order, 1e4, top)
    case = dict(op=op, bp=bp, order=order, ex=ex, ey=ey, ez=ez, arith=arith)
    if op == "solve":
        case.update(tol=0.0, iters=rng.choice([20, 35, 50]))
    return case


# ---- the mesh and its 1D rules ---------------------------------------------------------------

def _gll(n):
    """Gauss-Lobatto-Legendre nodes and weights, n points, in [-1, 1]."""
    c = np.zeros(n)
    c[-1] = 1.0
    leg = np.polynomial.legendre
    x = np.concatenate(([-1.0], np.sort(np.real(leg.legroots(leg.legder(c)))), [1.0]))
    d1, d2 = leg.legder(c), leg.legder(c, 2)
    for _ in range(3):  # Newton on P'
        x[1:-1] -= leg.legval(x[1:-1], d1) / leg.legval(x[1:-1], d2)
    x = 0.5 * (x - x[::-1])
    return x, 2.0 / (n * (n - 1) * leg.legval(x, c) ** 2)


def _bary(x):
    return np.array([1.0 / np.prod(x[i] - np.delete(x, i)) for i in range(len(x))])


def _interp(x, y):
    """Lagrange interpolation matrix from nodes x to points y."""
    b, out = _bary(x), np.zeros((len(y), len(x)))
    for r, t in enumerate(y):
        d = t - x
        hit = np.argmin(np.abs(d))
        if d[hit] == 0.0:
            out[r, hit] = 1.0
        else:
            out[r] = b / d / np.sum(b / d)
    return out


def _deriv(x):
    """Derivative matrix of the Lagrange basis on its own nodes."""
    b, n = _bary(x), len(x)
    D = np.zeros((n, n))
    for i in range(n):
        for j in range(n):
            if i != j:
                D[i, j] = b[j] / b[i] / (x[i] - x[j])
        D[i, i] = -np.sum(D[i])
    return D


def _axis(ne, order, dev):
    """Node positions of one direction, [ne, order + 1], and their global indices."""
    g = torch.from_numpy(0.5 * (_gll(order + 1)[0] + 1.0)).to(dev)
    e = torch.arange(ne, device=dev)
    return (e[:, None] + g[None, :]) / ne, e[:, None] * order + torch.arange(order + 1, device=dev)[None, :]


def _mesh(case, amp=AMP, dev="cuda"):
    """Deformed unit cube: coords [E, p1^3, 3], l2g [E, p1^3], Dirichlet flags [n]; i fastest, then j, k."""
    N, dims = case["order"], (case["ex"], case["ey"], case["ez"])
    p3 = (N + 1) ** 3
    (x, gx), (y, gy), (z, gz) = (_axis(n, N, dev) for n in dims)

    def spread(a, d):  # values of one direction over [ez, ey, ex, k, j, i]
        shape = [1] * 6
        shape[2 - d], shape[5 - d] = a.shape
        return a.reshape(shape).expand(dims[2], dims[1], dims[0], N + 1, N + 1, N + 1)

    X = [spread(a, d) for d, a in enumerate((x, y, z))]
    bump = amp * torch.sin(math.pi * X[0]) * torch.sin(math.pi * X[1]) * torch.sin(math.pi * X[2])
    coords = torch.stack([c + bump for c in X], -1).reshape(-1, p3, 3)
    nx, ny, nz = (N * n + 1 for n in dims)
    l2g = (spread(gx, 0) + nx * (spread(gy, 1) + ny * spread(gz, 2))).reshape(-1, p3)
    edge = torch.zeros(nz, ny, nx, dtype=torch.uint8, device=dev)
    edge[0], edge[-1], edge[:, 0], edge[:, -1], edge[:, :, 0], edge[:, :, -1] = 1, 1, 1, 1, 1, 1
    return coords, l2g, edge.reshape(-1)


def _host(mesh):
    return tuple(t.cpu().numpy() for t in mesh)


# ---- inputs ----------------------------------------------------------------------------------

def _rand(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * 2.0 - 1.0


def _ncomp(bp):
    return 3 if bp in (2, 4, 6) else 1


def _field(coords, seed):
    """kappa = exp(g) at the nodes, g a sum of 16 Fourier modes."""
    r = np.random.default_rng(seed)
    g = torch.zeros(coords.shape[:2], dtype=torch.float64, device=coords.device)
    for _ in range(16):
        k = [int(v) for v in r.integers(1, 5, 3)]
        a, ph = float(r.uniform(-0.125, 0.125)), [float(v) for v in r.uniform(0, 2 * math.pi, 3)]
        g += a * torch.cos(math.pi * k[0] * coords[..., 0] + ph[0]) * torch.cos(
            math.pi * k[1] * coords[..., 1] + ph[1]) * torch.cos(math.pi * k[2] * coords[..., 2] + ph[2])
    return torch.exp(g)


def _members(case, seed):
    """The independent problems of a batch: (order, elements per direction, deformation amplitude)."""
    r = np.random.default_rng(7 * case["problems"] + case["kmax"])  # the sizes belong to the case
    out = []
    for _ in range(case["problems"]):
        k = int(round(math.exp(r.uniform(math.log(case["kmin"]), math.log(case["kmax"])))))
        out.append((int(r.choice([3, 5, 7])), k, float(r.uniform(0.0, 0.1))))
    return out


def _member_case(order, k):
    return dict(op="solve", bp=5, order=order, ex=k, ey=k, ez=k)


def prepare(case, seed):
    if case["op"] == "batch":
        problems, bs = [], []
        for m, (order, k, amp) in enumerate(_members(case, seed)):
            coords, l2g, dirichlet = _mesh(_member_case(order, k), amp)
            bs.append(_rand(dirichlet.numel(), 1000 * seed + m) * (1 - dirichlet))
            problems.append((order,) + _host((coords, l2g, dirichlet)))
        return dict(case=case, batch=ceedbp.Batch(problems, arith=case["arith"]), bs=bs)
    mesh = _mesh(case)
    nc = _ncomp(case["bp"])
    op = ceedbp.Operator(case["bp"], case["order"], *_host(mesh), arith=case["arith"])
    n = mesh[2].numel()
    if case["op"] == "bk":
        shape = tuple(mesh[1].shape) + ((nc,) if nc == 3 else ())
        return dict(case=case, op=op, u=_rand(mesh[1].numel() * nc, seed).reshape(shape))
    if case["op"] == "adjoint":
        free = (1 - mesh[2]).double()
        b = op.mass(torch.ones_like(free)) * free
        op.set_kappa(_field(mesh[0], 2 * seed + 1))
        u_star, _ = op.solve(b, tol=1e-10)
        return dict(case=case, op=op, b=b, u_star=u_star, kappa=_field(mesh[0], 2 * seed))
    u = _rand(n * nc, seed).reshape((n, 3) if nc == 3 else (n,))
    if case["op"] == "apply":
        return dict(case=case, op=op, u=u)
    b = op.mass(u)
    if case["bp"] not in (1, 2):
        free = (1 - mesh[2]).double()
        b = b * (free[:, None] if nc == 3 else free)
    if case["op"] == "mixed":
        op.prepare_mixed(ceedbp.MIXED_FP32 if case["precision"] == "fp32" else ceedbp.MIXED_BF16)
    return dict(case=case, op=op, b=b)


def run(state):
    case, kind = state["case"], state["case"]["op"]
    if kind == "batch":
        xs, _ = state["batch"].solve(state["bs"], tol=1e-8)
        return xs
    op = state["op"]
    if kind == "apply":
        return op.apply(state["u"])
    if kind == "bk":
        return op.bk_apply(state["u"])
    if kind == "mixed":
        x, _ = op.solve(state["b"], tol=1e-10,
                        mixed=ceedbp.MIXED_FP32 if case["precision"] == "fp32" else ceedbp.MIXED_BF16)
        return x
    if kind == "adjoint":
        kappa = state["kappa"].detach().requires_grad_()
        J = ceedbp.kappa_misfit(kappa, op, state["b"], state["u_star"], tol=1e-10)
        J.backward()
        return {"J": J.detach(), "grad": kappa.grad}
    if case["iters"]:
        x, info = op.solve(state["b"], fixed_iters=case["iters"])
    else:
        x, info = op.solve(state["b"], tol=case["tol"])
    return x


# ---- what a pass cannot do without ---------------------------------------------------------------

def _flops_elem(bp, order):
    """Multiply-adds counted as two, of one component's element operator (the bake-off's own counts)."""
    p, q = order + 1, (order + 1 if bp in (5, 6) else order + 2)
    if bp in (5, 6):
        return 12 * p ** 4 + 15 * p ** 3
    interp = 4 * (p ** 3 * q + p ** 2 * q ** 2 + p * q ** 3)  # to the quadrature points and back
    return interp + q ** 3 if bp in (1, 2) else interp + 12 * q ** 4 + 15 * q ** 3


def _apply_work(case):
    bp, N = case["bp"], case["order"]
    E, nc, p = case["ex"] * case["ey"] * case["ez"], _ncomp(bp), N + 1
    q = p if bp in (5, 6) else p + 1
    n = (N * case["ex"] + 1) * (N * case["ey"] + 1) * (N * case["ez"] + 1)
    factors = 8 * E * q ** 3 * (1 if bp in (1, 2) else 6) + 4 * E * p ** 3
    return n * nc, E * p ** 3 * nc, factors, E * nc * _flops_elem(bp, N)


def _iteration_work(case):
    """One CG iteration: factors and map read once, x, r, p read and written, dinv read."""
    n, _, factors, flops = _apply_work(case)
    return factors + 8 * 7 * n, flops + 13 * n


def work(case):
    kind = case["op"]
    if kind == "batch":
        total = [0, 0]
        for order, k, _ in _members(case, 0):
            b, f = _iteration_work(_member_case(order, k))
            its = 10 + 4 * order * k  # CG iterations grow with the nodes per direction
            total[0] += b * its
            total[1] += f * its
        return dict(bytes=total[0], flops=total[1])
    if kind in ("apply", "bk"):
        n, nloc, factors, flops = _apply_work(case)
        if kind == "bk":
            p3 = (case["order"] + 1) ** 3 * case["ex"] * case["ey"] * case["ez"]
            return dict(bytes=factors - 4 * p3 + 16 * nloc, flops=flops)
        return dict(bytes=factors + 16 * n, flops=flops)
    b, f = _iteration_work(case)
    nodes = case["order"] * max(case["ex"], case["ey"], case["ez"])
    if kind == "mixed":
        its = 40 + 6 * nodes  # inner iterations; factors and vectors at the inner width
        return dict(bytes=b * its // (2 if case["precision"] == "fp32" else 3), flops=f * its)
    its = case.get("iters") or (20 + 4 * nodes)
    if kind == "adjoint":
        its *= 2
    return dict(bytes=b * its, flops=f * its)


# ---- 64-bit reference ------------------------------------------------------------------------------

class _Plain:
    """The bake-off operator by dense 1D contractions in torch float64."""

    def __init__(self, case, mesh, kappa=None):
        self.bp, N = case["bp"], case["order"]
        coords, self.l2g, dirichlet = mesh
        dev = coords.device
        p = N + 1
        x, w = _gll(p)
        if self.bp in (5, 6):
            self.J, D, wq, q = None, _deriv(x), w, p
        else:
            q = N + 2
            y, wq = np.polynomial.legendre.leggauss(q)
            self.J, D = torch.from_numpy(_interp(x, y)).to(dev), _deriv(y)
        self.p, self.q, self.n = p, q, dirichlet.numel()
        self.D = torch.from_numpy(D).to(dev)
        self.free = None if self.bp in (1, 2) else (1 - dirichlet).double()
        wq = torch.from_numpy(wq).to(dev)
        w3 = wq[:, None, None] * wq[None, :, None] * wq[None, None, :]
        X = [self.up(coords[..., d].reshape(-1, p, p, p)) for d in range(3)]
        jac = [self.grad(c) for c in X]  # jac[d][m] = d x_d / d r_m
        cof = [[None] * 3 for _ in range(3)]
        for d in range(3):
            for m in range(3):
                a, b, c, e = (d + 1) % 3, (d + 2) % 3, (m + 1) % 3, (m + 2) % 3
                cof[m][d] = jac[a][c] * jac[b][e] - jac[a][e] * jac[b][c]
        det = sum(jac[0][m] * cof[m][0] for m in range(3))
        self.mass_q = w3 * det
        if self.bp not in (1, 2):
            scale = w3 / det
            self.Ghat = {(a, b): scale * sum(cof[a][d] * cof[b][d] for d in range(3)) for a in range(3) for b in range(a, 3)}
            k = 1.0 if kappa is None else kappa.reshape(det.shape)
            self.G = {ab: g * k for ab, g in self.Ghat.items()}
        del jac, cof, X

    def up(self, u):  # nodes -> quadrature points, [E, k, j, i]
        if self.J is None:
            return u
        u = torch.matmul(u, self.J.T)
        u = torch.matmul(self.J, u)
        return torch.einsum("qk,ekji->eqji", self.J, u)

    def down(self, v):
        if self.J is None:
            return v
        v = torch.einsum("qk,eqji->ekji", self.J, v)
        v = torch.matmul(self.J.T, v)
        return torch.matmul(v, self.J)

    def grad(self, v):
        E, q = v.shape[0], self.q
        return (torch.matmul(v, self.D.T), torch.matmul(self.D, v),
                torch.matmul(self.D, v.reshape(E, q, q * q)).reshape(v.shape))

    def grad_t(self, f):
        E, q = f[0].shape[0], self.q
        return (torch.matmul(f[0], self.D) + torch.matmul(self.D.T, f[1]) +
                torch.matmul(self.D.T, f[2].reshape(E, q, q * q)).reshape(f[0].shape))

    def local(self, uL):  # [E, p^3] -> [E, p^3]
        p, out = self.p, torch.empty_like(uL)
        step = max(1, (1 << 22) // self.q ** 3)
        for e in range(0, uL.shape[0], step):
            s = slice(e, e + step)
            v = self.up(uL[s].reshape(-1, p, p, p))
            if self.bp in (1, 2):
                v = self.mass_q[s] * v
            else:
                g = self.grad(v)
                v = self.grad_t([sum(self.G[min(a, b), max(a, b)][s] * g[b] for b in range(3)) for a in range(3)])
            out[s] = self.down(v).reshape(-1, p ** 3)
        return out

    def sum_up(self, wL):
        return torch.zeros(self.n, dtype=torch.float64, device=wL.device).index_add_(0, self.l2g.reshape(-1), wL.reshape(-1))

    def masked(self, v):
        return v if self.free is None else v * self.free

    def apply(self, u):
        return self.masked(self.sum_up(self.local(self.masked(u)[self.l2g])))

    def mass(self, u):
        p, q = self.p, self.q
        v = self.up(u[self.l2g].reshape(-1, p, p, p)) * self.mass_q
        return self.sum_up(self.down(v).reshape(-1, p ** 3))

    def diagonal(self):
        """Diagonal of the assembled operator, by squared 1D tables."""
        J = torch.eye(self.p, dtype=torch.float64, device=self.D.device) if self.J is None else self.J
        if self.bp in (1, 2):
            terms = [(self.mass_q, (J * J,) * 3)]
        else:
            B = self.D @ J
            F = lambda a, d: B if a == d else J
            terms = [((1.0 if a == b else 2.0) * g, tuple(F(a, d) * F(b, d) for d in range(3))) for (a, b), g in self.G.items()]
        out = torch.zeros(self.l2g.shape, dtype=torch.float64, device=self.D.device)
        for g, (ti, tj, tk) in terms:
            v = torch.einsum("qk,eqji->ekji", tk, g)
            v = torch.matmul(tj.T, v)
            out += torch.matmul(v, ti).reshape(out.shape)
        return self.sum_up(out)

    def cg(self, b, iters=0, tol=0.0):
        dinv = self.masked(1.0 / self.diagonal())
        x, r = torch.zeros_like(b), b.clone()
        p = dinv * r
        rz, stop = torch.dot(r, p), (tol * torch.linalg.norm(b)).item()
        for it in range(iters or 20000):
            ap = self.apply(p)
            alpha = rz / torch.dot(p, ap)
            x += alpha * p
            r -= alpha * ap
            if not iters and it % 8 == 7 and torch.linalg.norm(r).item() <= stop:
                break
            z = dinv * r
            new = torch.dot(r, z)
            p = z + (new / rz) * p
            rz = new
        return x


def _columns(f, v):
    """f on each component of a vector field."""
    return f(v) if v.dim() == 1 else torch.stack([f(v[:, c].contiguous()) for c in range(3)], 1)


def exact(case, seed):
    if case["op"] == "batch":
        out = []
        for m, (order, k, amp) in enumerate(_members(case, seed)):
            mc = _member_case(order, k)
            mesh = _mesh(mc, amp)
            out.append(_Plain(mc, mesh).cg(_rand(mesh[2].numel(), 1000 * seed + m) * (1 - mesh[2]), tol=1e-12))
        return out
    mesh = _mesh(case)
    nc, n = _ncomp(case["bp"]), mesh[2].numel()
    if case["op"] == "adjoint":
        A = _Plain(case, mesh, _field(mesh[0], 2 * seed + 1))
        b = A.masked(A.mass(torch.ones(n, dtype=torch.float64, device="cuda")))
        u_star = A.cg(b, tol=1e-13)
        A = _Plain(case, mesh, _field(mesh[0], 2 * seed))
        u = A.cg(b, tol=1e-13)
        rhs = A.masked(A.mass(u - u_star))
        lam = A.cg(rhs, tol=1e-13)
        p = A.p
        gu, gl = (A.grad(v[mesh[1]].reshape(-1, p, p, p)) for v in (u, lam))
        g = -sum(A.Ghat[min(a, c), max(a, c)] * gl[a] * gu[c] for a in range(3) for c in range(3))
        return {"J": 0.5 * torch.dot(u - u_star, A.mass(u - u_star)), "grad": g.reshape(-1, p ** 3)}
    A = _Plain(case, mesh)
    if case["op"] == "bk":
        uL = _rand(mesh[1].numel() * nc, seed).reshape(tuple(mesh[1].shape) + ((nc,) if nc == 3 else ()))
        return A.local(uL) if nc == 1 else torch.stack([A.local(uL[..., c].contiguous()) for c in range(3)], 2)
    u = _rand(n * nc, seed).reshape((n, 3) if nc == 3 else (n,))
    if case["op"] == "apply":
        return _columns(A.apply, u)
    if case["op"] == "mixed":
        return _columns(lambda v: A.cg(A.masked(A.mass(v)), tol=1e-12), u)
    tol = 0.0 if case["iters"] else 1e-12
    return _columns(lambda v: A.cg(A.masked(A.mass(v)), iters=case["iters"], tol=tol), u)
