"""The work a user of this package has it do, as measurable cases.

Every case names one call through the public Python interface on one problem:

  operator   y = K x                             (StokesMG.vmult)
  smoothing  x <- S^2 (x, b)                     (StokesMG.smooth)
  cycle      x = MG(0, b)                        (StokesMG.vcycle)
  solve      FGMRES around the cycle             (StokesMG.solve)
  batch      independent meshes solved together  (StokesBatch.solve)
  gradient   solve and adjoint gradients         (stokes_solve_fn and backward)

Meshes are boxes of n = (nx, ny[, nz]) cells, coarsened while every count stays even and at least
four; "warped" moves the vertices by a smooth field of a tenth of a cell (general trilinear cells),
otherwise the cells are Cartesian.  "channel" is the box [0,4] x [0,1]^2 with an open outflow face.
The sizes are those of the package's benchmark and tests: the 2D 16^2 and 128^2 problems, the warped
cube of 32^3 cells, the Q3 channel, batches of uneven meshes, per-cell viscosities.

exact() is a plain 64-bit restatement: element matrices by quadrature, dense products per cell,
index_add, and the same multigrid written out on top of them.
"""
import math

import numpy as np
import torch

from paper_2205_15770_gb300 import ALL_FACES, StokesBatch, StokesMG, stokes_solve_fn

F64, F32 = "float64", "float32"


def listed():
    return [
        # a small 2D problem's operator: the smallest call, launches and latency
        dict(name="operator 2d 16^2 f64", kind="operator", n="16,16", k=2, dtype=F64, mesh="box"),
        # the operator of the general 3D problem, in the cycle's and in the outer loop's precision
        dict(name="operator 32^3 warped f32", kind="operator", n="32,32,32", k=2, dtype=F32, mesh="warped"),
        dict(name="operator 32^3 warped f64", kind="operator", n="32,32,32", k=2, dtype=F64, mesh="warped"),
        # a large flow problem on Cartesian cells: Q3, 23.7 million unknowns
        dict(name="operator 64^3 q3 channel f32", kind="operator", n="64,64,64", k=3, dtype=F32, mesh="channel"),
        # two smoothing steps as a caller's own cycle takes them, an inner level and a ragged box
        dict(name="smoothing 16^3 warped f32", kind="smoothing", n="16,16,16", k=2, dtype=F32, mesh="warped"),
        dict(name="smoothing 20x24x12 f64", kind="smoothing", n="20,24,12", k=2, dtype=F64, mesh="box"),
        # one preconditioner application: the general 3D problem, a ragged box in full precision, 2D
        dict(name="cycle 32^3 warped f32", kind="cycle", n="32,32,32", k=2, dtype=F32, mesh="warped"),
        dict(name="cycle 24x16x8 f64", kind="cycle", n="24,16,8", k=2, dtype=F64, mesh="box"),
        dict(name="cycle 2d 128^2 f32", kind="cycle", n="128,128", k=2, dtype=F32, mesh="box"),
        # a whole solve: implicit time step on the general 3D problem, cycle in f32, outer loop in f64
        dict(name="solve 32^3 warped", kind="solve", n="32,32,32", k=2, gamma=100.0, mesh="warped", cycle=F32),
        # several users' meshes of uneven size at once
        dict(name="batch 8,16,24,12", kind="batch", n="8;16;24;12", k=2, mesh="box", cycle=F32),
        # an inverse problem's step: new viscosities, forward and adjoint solve, both gradients
        dict(name="gradient 16^3", kind="gradient", n="16,16,16", k=2, mesh="box", cycle=F64),
    ]


def draw(rng):
    known = [{key: v for key, v in c.items() if key != "name"} for c in listed()]
    while (case := _draw(rng)) in known:
        pass
    return case


def _draw(rng):
    kind = rng.choice(["operator"] * 4 + ["smoothing"] * 3 + ["cycle"] * 4 + ["solve"] * 3 + ["batch"] + ["gradient"])
    two = rng.random() < 0.25

    def cells(lo, hi, dim, coarse=(2, 3, 5)):
        # coarsest counts of 2, 3 or 5 cells an axis, refined j times: near a size spread over the logarithm
        want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        j = max(1, round(math.log2(want / 3)))
        fits = [c << i for i in (j - 1, j, j + 1) if i >= 1 for c in coarse if lo <= c << i <= hi]
        size = min(fits, key=lambda v: abs(math.log(v / want)))
        j = next(i for i in range(1, 9) if size % (1 << i) == 0 and size >> i in coarse)
        fits = [c << j for c in coarse if lo <= c << j <= hi]
        return [size] * dim if rng.random() < 0.3 else [rng.choice(fits) for _ in range(dim)]

    def box(lo, hi, dim, coarse=(2, 3, 5)):
        return ",".join(map(str, cells(lo, hi, dim, coarse)))

    mesh = rng.choice(["warped", "box"])
    if kind == "operator":
        k = rng.choice([2, 2, 2, 3, 4])
        if two:
            n = box(12, 256, 2)
        else:
            n = box(8, {2: 64, 3: 32, 4: 16}[k], 3, {2: (2, 3, 5), 3: (2, 3), 4: (2,)}[k])
            mesh = rng.choice([mesh, "channel"])
        return dict(kind=kind, n=n, k=k, dtype=rng.choice([F32, F64]), mesh=mesh)
    if kind in ("smoothing", "cycle"):
        return dict(kind=kind, n=box(12, 192, 2) if two else box(8, 40, 3), k=2, dtype=rng.choice([F32, F32, F64]), mesh=mesh)
    if kind == "solve":
        return dict(kind=kind, n=box(12, 96, 2) if two else box(8, 32, 3), k=2, gamma=rng.choice([0.0, 100.0, 1e4]), mesh=mesh,
                    cycle=rng.choice([F32, F32, F64]))
    if kind == "batch":
        return dict(kind=kind, n=";".join(str(cells(8, 24, 1)[0]) for _ in range(rng.randint(2, 5))), k=2, mesh="box", cycle=F32)
    return dict(kind=kind, n=box(8, 16, 3), k=2, mesh="box", cycle=F64)


# ---- problem data ------------------------------------------------------------------------------

def _counts(text):
    return tuple(int(v) for v in text.split(","))


def _levels(n):
    """Coarsen while every count is even and leaves at least two cells."""
    levels = 1
    while all(v % 2 == 0 and v >= 4 for v in n):
        n, levels = tuple(v // 2 for v in n), levels + 1
    return levels


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _warp(n, seed):
    """Vertices of the unit box moved by up to a tenth of a cell along a smooth field that vanishes on the boundary."""
    rng = np.random.default_rng(seed)
    d = len(n)
    ax = [np.linspace(0.0, 1.0, v + 1) for v in n]
    X = np.stack(np.meshgrid(*ax[::-1], indexing="ij")[::-1], axis=-1)
    bubble = np.prod(np.sin(np.pi * X), axis=-1)
    V = X.copy()
    for c in range(d):
        wave = sum(np.sin(2 * np.pi * (X @ rng.integers(0, 3, size=d)) + rng.uniform(0, 2 * np.pi)) for _ in range(3)) / 3
        V[..., c] += 0.1 / n[c] * bubble * wave
    return V


def _options(case, seed):
    """Arguments of StokesMG for a case's mesh: the recommended smoother, two steps with one Chebyshev step each."""
    n = _counts(case["n"])
    dim = len(n)
    o = dict(dim=dim, n=n, n_levels=_levels(n), k=case["k"], gamma_rho=case.get("gamma", 0.0), kA=1, kS=1, m=2,
             schur_diag="d" if case["k"] == 2 else "loc")
    if case["mesh"] == "warped":
        o["vertices"] = _warp(n, seed)
    elif case["mesh"] == "channel":
        o.update(hi=(4.0, 1.0, 1.0), dirichlet_faces=ALL_FACES[3] & ~0x2, mu=1e-3)
    if case.get("cycle") == F64:
        o["vcycle_fp32"] = False
    return o


def _sizes(n, k):
    nv, npr = math.prod(k * v + 1 for v in n), math.prod((k - 1) * v + 1 for v in n)
    return len(n) * nv, npr


def _free(n, k, faces):
    """Mask over the velocity nodes: True where no Dirichlet face holds the node."""
    m = torch.ones(tuple(k * v + 1 for v in n[::-1]), dtype=torch.bool, device="cuda")
    for a in range(len(n)):
        axis = len(n) - 1 - a
        if faces >> (2 * a) & 1:
            m.index_fill_(axis, torch.tensor([0], device="cuda"), False)
        if faces >> (2 * a + 1) & 1:
            m.index_fill_(axis, torch.tensor([k * n[a]], device="cuda"), False)
    return m.reshape(-1)


def _vector(n, k, seed):
    n_u, n_p = _sizes(n, k)
    return torch.rand(n_u + n_p, dtype=torch.float64, device="cuda", generator=_generator(seed)) * 2 - 1


def _residual(n, k, faces, seed):
    """A residual-like vector: random, zero at Dirichlet nodes, the pressure part of zero mean."""
    b = _vector(n, k, seed)
    n_u, _ = _sizes(n, k)
    b[:n_u] *= _free(n, k, faces).repeat(len(n))
    b[n_u:] -= b[n_u:].mean()
    return b


def _forcing(n, k, seed):
    """Four random Fourier modes per component on the velocity lattice."""
    rng = np.random.default_rng(seed)
    d = len(n)
    ax = [np.linspace(0.0, 1.0, k * v + 1) for v in n]
    f = np.zeros((d,) + tuple(len(a) for a in ax[::-1]))
    for c in range(d):
        for _ in range(4):
            term = rng.standard_normal()
            for a in range(d):
                s = np.sin(np.pi * rng.integers(1, 4) * ax[a])
                term = term * s.reshape([-1 if i == d - 1 - a else 1 for i in range(d)])
            f[c] += term
    return torch.as_tensor(f.reshape(-1), device="cuda")


def _viscosity(n, seed):
    """exp of a smooth random field, one value per cell."""
    rng = np.random.default_rng(seed)
    ax = [(np.arange(v) + 0.5) / v for v in n]
    X = np.stack(np.meshgrid(*ax[::-1], indexing="ij")[::-1], axis=-1)
    g = sum(rng.standard_normal() * np.cos(np.pi * (X @ rng.integers(0, 4, size=len(n))) + rng.uniform(0, 2 * np.pi)) for _ in range(6))
    return np.exp(0.5 * g).reshape(-1)


def _members(case):
    return [dict(case, n=",".join([c] * 3), gamma=1000.0 if i % 2 else 0.0) for i, c in enumerate(case["n"].split(";"))]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        members = _members(case)
        opts = [_options(m, seed + i) for i, m in enumerate(members)]
        shared = {key: opts[0].pop(key) for key in ("kA", "kS", "m", "schur_diag")}
        B = StokesBatch([{key: v for key, v in o.items() if key not in shared} for o in opts], **shared)
        bs = [M.mass_rhs(_forcing(o["n"], case["k"], seed + i)) for i, (M, o) in enumerate(zip(B.members, opts))]
        return {"kind": kind, "B": B, "bs": bs}
    o = _options(case, seed)
    n, k, faces = o["n"], o["k"], o.get("dirichlet_faces", ALL_FACES[o["dim"]])
    if kind == "gradient":
        mu = torch.as_tensor(_viscosity(n, seed), device="cuda").requires_grad_()
        f = _forcing(n, k, seed).requires_grad_()
        S = StokesMG(mu_cell=_viscosity(n, seed + 1), **o)  # last step's viscosities
        return {"kind": kind, "S": S, "mu": mu, "f": f, "seedling": _residual(n, k, faces, seed + 2)}
    S = StokesMG(**o)
    if kind == "solve":
        return {"kind": kind, "S": S, "b": S.mass_rhs(_forcing(n, k, seed))}
    dtype = getattr(torch, case["dtype"])
    if kind == "operator":
        return {"kind": kind, "S": S, "x": _vector(n, k, seed).to(dtype)}
    s = {"kind": kind, "S": S, "b": _residual(n, k, faces, seed).to(dtype)}
    if kind == "smoothing":
        s["x0"] = _residual(n, k, faces, seed + 1).to(dtype)
    return s


def run(state):
    kind = state["kind"]
    if kind == "operator":
        return state["S"].vmult(state["x"])
    if kind == "smoothing":
        return state["S"].smooth(state["b"], state["x0"].clone(), steps=2)
    if kind == "cycle":
        return state["S"].vcycle(state["b"])
    if kind == "solve":
        return state["S"].solve(state["b"], rtol=1e-8)[0]
    if kind == "batch":
        return state["B"].solve(state["bs"], rtol=1e-8)[0]
    mu, f = state["mu"].detach().requires_grad_(), state["f"].detach().requires_grad_()
    x = stokes_solve_fn(state["S"], mu, f, rtol=1e-10)
    x.backward(state["seedling"])
    return x.detach(), mu.grad, f.grad


# ---- what a pass cannot do without ---------------------------------------------------------------

def _flops(n, k, a=0, bt=0, b=0):
    """Sum-factorised flops of `a` applications of A, `bt` of B^T and `b` of B: 1D sweeps of two flops per term and the point operations."""
    d, q = len(n), k + 1
    grad = d * 2 * d * 2 * q ** (d + 1)              # values and gradients of d components
    pre = d * 2 * q ** d * k                         # pressure to or from the Gauss points
    per = a * (2 * grad + d * 2 * d * d * q ** d) + (bt + b) * (grad + pre + 2 * d * d * q ** d)
    return math.prod(n) * per


def _cycle_flops(n, k):
    """Two smoothing steps before and after, the residual, on every level but the coarsest."""
    total = 0
    while all(v % 2 == 0 and v >= 4 for v in n):
        total += _flops(n, k, a=15 + 1, bt=11 + 1, b=8 + 1)  # a zero first iterate saves one A + B^T
        n = tuple(v // 2 for v in n)
    return total + 2 * sum(_sizes(n, k)) ** 2


def work(case):
    if case["kind"] == "batch":
        parts = [work(dict(m, kind="solve")) for m in _members(case)]
        return {key: sum(p[key] for p in parts) for key in ("bytes", "flops")}
    n, k = _counts(case["n"]), case["k"]
    N, cells = sum(_sizes(n, k)), math.prod(n)
    size = 4 if case.get("dtype") == F32 else 8
    geometry = len(n) * math.prod(v + 1 for v in n) if case["mesh"] == "warped" else 0
    operator = _flops(n, k, a=1, bt=1, b=1)
    kind = case["kind"]
    if kind == "operator":
        return {"bytes": size * (2 * N + geometry), "flops": operator}
    if kind == "smoothing":  # b and x in, x out, the two diagonals
        return {"bytes": size * (4 * N + geometry), "flops": _flops(n, k, a=8, bt=6, b=4)}
    if kind == "cycle":
        return {"bytes": size * (3 * N + geometry), "flops": _cycle_flops(n, k)}
    # five iterations of a cycle and an operator are what this problem family takes
    solve = 5 * (_cycle_flops(n, k) + operator)
    if kind == "solve":
        return {"bytes": 8 * (2 * N + geometry), "flops": solve}
    return {"bytes": 8 * (4 * N + 4 * cells), "flops": 4 * solve}  # forward and adjoint, to 1e-10


# ---- the same in plain 64-bit arithmetic ------------------------------------------------------------

def _lagrange(nodes, x):
    """Values and derivatives of the Lagrange polynomials through `nodes` at x: (nodes, points) each."""
    c = np.polynomial.polynomial
    val, der = [], []
    for i, t in enumerate(nodes):
        p = np.ones(1)
        for j, s in enumerate(nodes):
            if j != i:
                p = c.polymul(p, np.array([-s, 1.0]) / (t - s))
        val.append(c.polyval(x, p))
        der.append(c.polyval(x, c.polyder(p)) if len(p) > 1 else np.zeros_like(x))
    return np.array(val), np.array(der)


def _lobatto(degree):
    inner = np.polynomial.legendre.Legendre.basis(degree).deriv().roots().real if degree > 1 else np.zeros(0)
    return np.concatenate([[0.0], (np.sort(inner) + 1) / 2, [1.0]])


def _tensor(mats):
    """Tensor product of 1D tables (functions, points), given for x, y[, z]; x fastest in both indices."""
    out = mats[0]
    for m in mats[1:]:
        out = np.kron(m, out)
    return torch.as_tensor(out, device="cuda")


class _Plain:
    """One level: element matrices by quadrature, products per cell, sums by index_add."""

    def __init__(self, n, k, mu=1.0, gamma_rho=0.0, vertices=None, hi=(1.0, 1.0, 1.0), faces=None, mu_cell=None):
        d = len(n)
        self.n, self.k, self.d = n, k, d
        self.faces = ALL_FACES[d] if faces is None else faces
        self.n_u, self.n_p = _sizes(n, k)
        self.nv = self.n_u // d
        self.free = _free(n, k, self.faces)
        self.pker = self.faces == ALL_FACES[d]
        gx, gw = np.polynomial.legendre.leggauss(k + 1)
        gx, gw = (gx + 1) / 2, gw / 2
        v, dv = _lagrange(_lobatto(k), gx)
        p, _ = _lagrange(_lobatto(k - 1), gx)
        g, dg = _lagrange([0.0, 1.0], gx)
        phi = _tensor([v] * d)
        dphi = torch.stack([_tensor([dv if a == b else v for b in range(d)]) for a in range(d)])
        psi = _tensor([p] * d)
        dgeo = torch.stack([_tensor([dg if a == b else g for b in range(d)]) for a in range(d)])
        w = _tensor([gw.reshape(1, -1)] * d).reshape(-1)
        if vertices is None:
            X = torch.as_tensor(np.stack(np.meshgrid(*[np.array([0.0, hi[a] / n[a]]) for a in range(d)][::-1], indexing="ij")[::-1], -1).reshape(1, 2 ** d, d), device="cuda")
        else:
            V = torch.as_tensor(np.ascontiguousarray(vertices), device="cuda").reshape(-1, d)
            X = V[self._nodes(n, 1)]
        self.vn, self.pn = self._nodes(n, k), self._nodes(n, k - 1)
        mus = torch.full((1,), float(mu), dtype=torch.float64, device="cuda") if mu_cell is None else torch.as_tensor(mu_cell, device="cuda")
        K, M, B = [], [], []
        for x in X.split(4096):
            J = torch.einsum("cva,bvq->cqab", x, dgeo)
            wd = torch.linalg.det(J) * w
            grad = torch.einsum("cqba,biq->caiq", torch.linalg.inv(J), dphi)
            K.append(torch.einsum("caiq,cajq->cij", grad * wd[:, None, None], grad))
            M.append(torch.einsum("cq,iq,jq->cij", wd, phi, phi))
            B.append(-torch.einsum("cq,iq,cajq->ciaj", wd, psi, grad))
        self.K0, self.M, self.B = torch.cat(K), torch.cat(M), torch.cat(B)
        self.A = mus[:, None, None] * self.K0 + gamma_rho * self.M

    def _nodes(self, n, k):
        """Lattice indices of every cell's nodes, both with x fastest."""
        N = [k * v + 1 for v in n]
        cell = local = torch.zeros(1, dtype=torch.int64, device="cuda")
        stride = 1
        for a in range(len(n)):
            cell = (k * torch.arange(n[a], device="cuda")[:, None] * stride + cell).reshape(-1)
            local = (torch.arange(k + 1, device="cuda")[:, None] * stride + local).reshape(-1)
            stride *= N[a]
        return cell[:, None] + local

    @staticmethod
    def _each(E, x):
        """Per-cell products of the element matrices (one for all cells, or one each) and vectors (cells, entries)."""
        return x @ E[0].T if E.shape[0] == 1 else torch.bmm(E, x[:, :, None])[:, :, 0]

    def _velocity(self, E, u, mask_in, mask_out):
        out = torch.zeros(self.d, self.nv, dtype=torch.float64, device="cuda")
        for c, uc in enumerate(u.view(self.d, self.nv)):
            uc = uc * self.free if mask_in else uc
            out[c].index_add_(0, self.vn.reshape(-1), self._each(E, uc[self.vn]).reshape(-1))
            if mask_out:
                out[c] *= self.free
        return out.reshape(-1)

    def apply_A(self, u):  # identity at Dirichlet nodes
        fixed = ~self.free.repeat(self.d)
        return self._velocity(self.A, u, True, True) + u * fixed

    def mass(self, u, mask_in=False, mask_out=True):
        return self._velocity(self.M, u, mask_in, mask_out)

    def apply_B(self, u):
        out = torch.zeros(self.n_p, dtype=torch.float64, device="cuda")
        for c, uc in enumerate(u.view(self.d, self.nv)):
            out.index_add_(0, self.pn.reshape(-1), self._each(self.B[:, :, c], (uc * self.free)[self.vn]).reshape(-1))
        return out

    def apply_BT(self, p):
        out = torch.zeros(self.d, self.nv, dtype=torch.float64, device="cuda")
        for c in range(self.d):
            out[c].index_add_(0, self.vn.reshape(-1), self._each(self.B[:, :, c].transpose(1, 2), p[self.pn]).reshape(-1))
            out[c] *= self.free
        return out.reshape(-1)

    def apply(self, x):
        u, p = x[:self.n_u], x[self.n_u:]
        return torch.cat([self.apply_A(u) + self.apply_BT(p), self.apply_B(u)])

    # -- smoother: diagonals, largest eigenvalues, one inexact Uzawa step
    def set_up(self, schur):
        d, nc = self.d, self.vn.shape[0]
        dA = torch.diagonal(self.A, dim1=1, dim2=2).expand(nc, -1)
        D = torch.zeros(self.nv, dtype=torch.float64, device="cuda").index_add_(0, self.vn.reshape(-1), dA.reshape(-1))
        D = torch.where(self.free, D, torch.ones_like(D))
        self.DA = D.repeat(d)
        self.DS = torch.zeros(self.n_p, dtype=torch.float64, device="cuda")
        if schur == "loc":
            f = self.free[self.vn].double() / dA
            loc = torch.einsum("ciaj,cj->ci", self.B.expand(nc, -1, -1, -1) ** 2, f)
            self.DS.index_add_(0, self.pn.reshape(-1), loc.reshape(-1))
        else:  # diag(B diag(A)^-1 B^T): the assembled entries of B, one component at a time
            rows = self.pn[:, :, None].expand(-1, -1, self.vn.shape[1]).reshape(-1)
            cols = self.vn[:, None, :].expand(-1, self.pn.shape[1], -1).reshape(-1)
            key, at = torch.unique(rows * self.nv + cols, return_inverse=True)
            for c in range(d):
                full = self.B[:, :, c].expand(nc, -1, -1).reshape(-1)
                val = torch.zeros(len(key), dtype=torch.float64, device="cuda").index_add_(0, at, full)
                self.DS.index_add_(0, key // self.nv, val ** 2 * (self.free / D)[key % self.nv])
        c1 = 3.0 * 2 * 3.0 - 1.0  # C_2(3)
        self.scale = c1 / (1 + c1)
        s = self.DA.rsqrt()
        v0 = _splitmix(0x5EED, self.n_u) * self.free.repeat(d)
        self.beta_A = 1.1 * _ritz(lambda v: s * self.apply_A(s * v), v0)
        t = self.DS.rsqrt()
        v0 = _splitmix(0x5EED + 1, self.n_p)
        if self.pker:
            z = self.DS.sqrt()
            v0 = v0 - (v0 @ z) / (z @ z) * z
        self.beta_S = 1.1 * _ritz(lambda v: t * self.schur(t * v), v0)

    def _chebyshev(self, apply, D, r, beta):  # one step, on [beta / 2, beta]
        theta, delta = 0.75 * beta, 0.25 * beta
        s1 = theta / delta
        x = r / D / theta
        rho = 1 / (2 * s1 - 1 / s1)
        return self.scale * (x + rho / s1 * x + 2 * rho / delta * (r - apply(x)) / D)

    def inverse_A(self, r):
        return self._chebyshev(self.apply_A, self.DA, r, self.beta_A)

    def schur(self, q):
        return self.apply_B(self.inverse_A(self.apply_BT(q)))

    def smooth(self, x, b, steps=2):
        u, p = x[:self.n_u], x[self.n_u:]
        f, g = b[:self.n_u], b[self.n_u:]
        for _ in range(steps):
            hat = u + self.inverse_A(f - self.apply_A(u) - self.apply_BT(p))
            dp = self._chebyshev(self.schur, self.DS, self.apply_B(hat) - g, self.beta_S)
            u, p = hat - self.inverse_A(self.apply_BT(dp)), p + dp
        return torch.cat([u, p])


def _splitmix(seed, n):
    i = np.arange(1, n + 1, dtype=np.uint64)
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + i * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return torch.as_tensor(2.0 * ((z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53) - 1.0, device="cuda")


def _ritz(apply, v0, steps=40):
    """Largest Ritz value of plain Lanczos."""
    v, last, b, al, be = v0 / v0.norm(), torch.zeros_like(v0), 0.0, [], []
    for j in range(steps):
        w = apply(v) - b * last
        a = float(w @ v)
        w = w - a * v
        al.append(a)
        b = float(w.norm())
        if j == steps - 1 or b <= 1e-14 * max(abs(a), 1.0):
            break
        be.append(b)
        last, v = v, w / b
    be = be[:len(al) - 1]
    return float(np.linalg.eigvalsh(np.diag(al) + np.diag(be, 1) + np.diag(be, -1))[-1])


class _PlainMG:
    """The multigrid cycle written out on _Plain levels."""

    def __init__(self, o, mu_cell=None, only_finest=False):
        n, k, top = o["n"], o["k"], o["n_levels"] - 1
        self.levels = []
        for l in ([top] if only_finest else range(top + 1)):
            s = 1 << (top - l)
            m = tuple(v // s for v in n)
            V = o.get("vertices")
            if V is not None:
                V = V[tuple(slice(None, None, s) for _ in n)]
            mc = mu_cell
            if mc is not None and s > 1:
                mc = mc.reshape([x for v in m[::-1] for x in (v, s)]).mean(axis=tuple(range(1, 2 * len(n), 2))).reshape(-1)
            self.levels.append(_Plain(m, k, o.get("mu", 1.0), o.get("gamma_rho", 0.0), V, o.get("hi", (1.0, 1.0, 1.0)), o.get("dirichlet_faces"), mc))
        if only_finest:
            return
        c = self.levels[0]
        E = torch.eye(c.n_u + c.n_p, dtype=torch.float64, device="cuda")
        K = torch.stack([c.apply(e) for e in E], 1)
        if c.pker:
            e = torch.cat([torch.zeros(c.n_u, device="cuda"), torch.ones(c.n_p, device="cuda")]).double()
            K = torch.cat([torch.cat([K, e[:, None]], 1), torch.cat([e, e.new_zeros(1)])[None]], 0)
        self.coarse = torch.linalg.inv(K)[:c.n_u + c.n_p, :c.n_u + c.n_p]
        for L in self.levels[1:]:
            L.set_up(o["schur_diag"])

    def _inject(self, l, x, down):
        """P x from level l - 1 to l, or P^T x from l to l - 1, axis by axis."""
        f, c = self.levels[l], self.levels[l - 1]
        src, dst = (f, c) if down else (c, f)
        out = []
        for comp in range(f.d + 1):
            vel = comp < f.d
            k = f.k if vel else f.k - 1
            y = x[comp * src.nv:(comp + 1) * src.nv] * src.free if vel else x[src.n_u:]
            y = y.view([k * v + 1 for v in src.n[::-1]])
            for a in range(f.d):
                P = _injection(k, c.n[a])
                y = torch.movedim(torch.tensordot(P.T if down else P, y, dims=([1], [f.d - 1 - a])), 0, f.d - 1 - a)
            out.append(y.reshape(-1) * dst.free if vel else y.reshape(-1))
        return torch.cat(out)

    def cycle(self, x, b, l=None):
        l = len(self.levels) - 1 if l is None else l
        if l == 0:
            return self.coarse @ b
        L = self.levels[l]
        x = L.smooth(x, b)
        r = self._inject(l, b - L.apply(x), True)
        x = x + self._inject(l, self.cycle(torch.zeros_like(r), r, l - 1), False)
        return L.smooth(x, b)

    def solve(self, b, reduction=1e-13):
        """Flexible GMRES, restarted until the residual stops at the reduction or at rounding."""
        x, L = torch.zeros_like(b), self.levels[-1]
        for _ in range(4):
            r = b - L.apply(x)
            if r.norm() <= reduction * b.norm():
                break
            V, Z, H = [r / r.norm()], [], np.zeros((21, 20))
            for j in range(20):
                Z.append(self.cycle(torch.zeros_like(b), V[-1]))
                w = L.apply(Z[-1])
                for _pass in range(2):
                    for i, v in enumerate(V):
                        h = float(w @ v)
                        H[i, j] += h
                        w = w - h * v
                H[j + 1, j] = float(w.norm())
                rhs = np.zeros(j + 2)
                rhs[0] = float(r.norm())
                y = np.linalg.lstsq(H[:j + 2, :j + 1], rhs, rcond=None)[0]
                if np.linalg.norm(rhs - H[:j + 2, :j + 1] @ y) <= reduction * float(b.norm()) or H[j + 1, j] == 0:
                    break
                V.append(w / w.norm())
            for z, c in zip(Z, y):
                x = x + float(c) * z
        if L.pker:
            x[L.n_u:] -= x[L.n_u:].mean()
        return x


def _injection(k, coarse):
    t = _lobatto(k)
    P = np.zeros((2 * k * coarse + 1, k * coarse + 1))
    for i in range(len(P)):
        f = min(i // k, 2 * coarse - 1)
        P[i, k * (f // 2):k * (f // 2) + k + 1] = _lagrange(t, np.array([(f % 2 + t[i - k * f]) / 2]))[0][:, 0]
    return torch.as_tensor(P, device="cuda")


def _solution(o, seed, k, mu_cell=None):
    mg = _PlainMG(o, mu_cell)
    return mg, mg.solve(torch.cat([mg.levels[-1].mass(_forcing(o["n"], k, seed)), torch.zeros(mg.levels[-1].n_p, dtype=torch.float64, device="cuda")]))


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [_solution(_options(m, seed + i), seed + i, case["k"])[1] for i, m in enumerate(_members(case))]
    o = _options(case, seed)
    n, k, faces = o["n"], o["k"], o.get("dirichlet_faces", ALL_FACES[o["dim"]])
    if kind == "operator":
        x = _vector(n, k, seed).to(getattr(torch, case["dtype"])).double()
        return _PlainMG(o, only_finest=True).levels[0].apply(x)
    if kind == "solve":
        return _solution(o, seed, k)[1]
    if kind == "gradient":
        mg, x = _solution(o, seed, k, _viscosity(n, seed))
        L = mg.levels[-1]
        lam = mg.solve(_residual(n, k, faces, seed + 2))
        gmu = 0
        for c in range(L.d):
            l, u = ((v[c * L.nv:(c + 1) * L.nv] * L.free)[L.vn] for v in (lam, x))
            gmu = gmu - (l * L._each(L.K0, u)).sum(1)
        return x, gmu, L.mass(lam[:L.n_u], mask_in=True, mask_out=False)
    dtype = getattr(torch, case["dtype"])
    b = _residual(n, k, faces, seed).to(dtype).double()
    mg = _PlainMG(o)
    if kind == "smoothing":
        return mg.levels[-1].smooth(_residual(n, k, faces, seed + 1).to(dtype).double(), b)
    return mg.cycle(torch.zeros_like(b), b)
