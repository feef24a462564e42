"""The fixed-point FP64 cell kernel (launch shape 5, k = 2): its error against extended precision is no larger
than the floating-point column kernel's, it agrees with that kernel block by block at the edges of its groups of
ten cells, and inputs outside its range (infinities, NaN, extreme exponents, zero parts) behave as there."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu
LD = np.longdouble


def _apply(n, V, x, mu_cell, grho):
    """K x of Q2-Q1 by plain quadrature in extended precision, every boundary velocity node constrained."""
    r = np.sqrt(LD(15)) / 10
    g, w = np.array([LD(1) / 2 - r, LD(1) / 2, LD(1) / 2 + r]), np.array([LD(5), LD(8), LD(5)]) / 18
    val = np.array([[2 * t * t - 3 * t + 1, 4 * t - 4 * t * t, 2 * t * t - t] for t in g])
    der = np.array([[4 * t - 3, 4 - 8 * t, 4 * t - 1] for t in g])
    lin, dlin = np.array([[1 - t, t] for t in g]), np.array([[LD(-1), LD(1)]] * 3)

    def tensor(a, b, c):  # rows: points, columns: functions, x fastest in both
        return np.einsum("ai,bj,ck->cbakji", a, b, c).reshape(27, -1)

    phi, psi = tensor(val, val, val), tensor(lin, lin, lin)
    D = [tensor(der, val, val), tensor(val, der, val), tensor(val, val, der)]
    G = [tensor(dlin, lin, lin), tensor(lin, dlin, lin), tensor(lin, lin, dlin)]
    wt = np.einsum("c,b,a->cba", w, w, w).reshape(-1)
    N = [2 * v + 1 for v in n]
    nu = 3 * N[0] * N[1] * N[2]
    full = x[:nu].reshape(3, N[2], N[1], N[0])
    free = np.zeros(full.shape, dtype=bool)
    free[:, 1:-1, 1:-1, 1:-1] = True
    u, p = np.where(free, full, LD(0)), x[nu:].reshape(n[2] + 1, n[1] + 1, n[0] + 1)
    yu, yp = np.zeros_like(u), np.zeros_like(p)
    mu_cell = mu_cell.reshape(n[::-1])
    for cz, cy, cx in np.ndindex(*n[::-1]):
        X = V[cz:cz + 2, cy:cy + 2, cx:cx + 2].reshape(8, 3)
        J = [t @ X for t in G]
        adj = np.stack([np.cross(J[1], J[2]), np.cross(J[2], J[0]), np.cross(J[0], J[1])], 1)
        det = (J[0] * adj[:, 0]).sum(1)
        su = (slice(2 * cz, 2 * cz + 3), slice(2 * cy, 2 * cy + 3), slice(2 * cx, 2 * cx + 3))
        sp = (slice(cz, cz + 2), slice(cy, cy + 2), slice(cx, cx + 2))
        pq, qa = psi @ p[sp].reshape(-1), np.zeros(27, LD)
        for c in range(3):
            uc = u[(c,) + su].reshape(-1)
            ref = np.stack([d @ uc for d in D], 1)
            phys = np.einsum("qba,qb->qa", adj, ref) / det[:, None]
            f = np.einsum("qba,qa->qb", adj, phys) * (mu_cell[cz, cy, cx] * wt)[:, None] - (pq * wt)[:, None] * adj[:, :, c]
            y = sum(D[b].T @ f[:, b] for b in range(3)) + phi.T @ (grho * wt * det * (phi @ uc))
            yu[(c,) + su] += y.reshape(3, 3, 3)
            qa -= wt * (adj[:, :, c] * ref).sum(1)
        yp[sp] += (psi.T @ qa).reshape(2, 2, 2)
    return np.concatenate([np.where(free, yu, full).reshape(-1), yp.reshape(-1)]), nu


def _solver(n, warped, seed=1, stretch=(1.0, 1.0, 1.0), **kw):
    from paper_2205_15770_gb300 import StokesMG
    V = (W.perturbed_vertices(3, n, seed=seed) if warped else W.lattice_vertices(3, n)) * np.array(stretch)
    S = StokesMG(dim=3, n=n, n_levels=1, k=2, vertices=V if warped else None, hi=stretch, **kw)
    return S, V


def _both(S, f):
    out = []
    for shape in (5, 4):
        S.set_launch_shape(0, shape, 64)
        out.append(f())
    return out


@pytest.mark.parametrize("field", ["random", "smooth", "large pressure"])
@pytest.mark.parametrize("case", [
    dict(n=(4, 4, 4), warped=True), dict(n=(4, 3, 2), warped=True, gamma_rho=1e4, mu=1e-3),
    dict(n=(4, 3, 2), warped=False, gamma_rho=100.0), dict(n=(3, 4, 2), warped=False, stretch=(1.0, 0.1, 20.0)),
    dict(n=(3, 2, 4), warped=False, cells=True, gamma_rho=1.0), dict(n=(3, 2, 4), warped=True, cells=True)])
def test_error_is_no_larger_than_in_floating_point(case, field):
    kw = dict(case)
    n, cells = kw["n"], kw.pop("cells", False)
    rng = np.random.default_rng(3)
    mu = rng.uniform(0.1, 10.0, int(np.prod(n))) if cells else np.full(int(np.prod(n)), kw.get("mu", 1.0))
    S, V = _solver(mu_cell=mu if cells else None, **kw)
    x = rng.uniform(-1, 1, S.size())
    nu = S.sizes()[0]
    if field == "smooth":
        z, y, xx = np.meshgrid(*[np.linspace(0, 1, 2 * v + 1) for v in n[::-1]], indexing="ij")
        s = (np.sin(np.pi * xx) * np.sin(np.pi * y) * np.sin(np.pi * z)).reshape(-1)
        x[:nu] = np.concatenate([s, 2 * s, 3 * s])
    elif field == "large pressure":
        x[nu:] *= 1e9
    ref, _ = _apply(n, V.astype(LD), x.astype(LD), mu.astype(LD), LD(kw.get("gamma_rho", 0.0)))
    t = torch.as_tensor(x, device="cuda")
    y5, y4 = _both(S, lambda: S.vmult(t).cpu().numpy())
    for part in (slice(0, nu), slice(nu, None)):
        scale = np.linalg.norm(ref[part].astype(float))
        e5, e4 = (np.linalg.norm((y - ref)[part].astype(float)) / scale for y in (y5, y4))
        # one rounding to FP64 per cell's contribution and per sum stays in either form: 2^-53 times at most 8
        assert e5 <= max(e4, 2.0 ** -51), (e5, e4)


@pytest.mark.parametrize("n", [(1, 1, 1), (1, 1, 10), (3, 5, 7), (11, 2, 1)])
@pytest.mark.parametrize("warped", [False, True])
def test_blocks_match_the_column_kernel(n, warped):
    S, _ = _solver(n, warped, gamma_rho=10.0, dirichlet_faces=0x3F & ~0x2)
    nu, npr = S.sizes()
    rng = np.random.default_rng(5)
    u, p = (torch.as_tensor(rng.uniform(-1, 1, m), device="cuda") for m in (nu, npr))
    for blocks in (1, 2, 4, 3, 7):
        (au, ap), (bu, bp) = _both(S, lambda: S.apply_blocks(blocks, u=u if blocks & 5 else None, p=p if blocks & 2 else None))
        for a, b in ((au, bu), (ap, bp)):
            if a is not None:  # two FP64 results of sums of up to 8 cells: a few roundings of the largest entry
                assert (a - b).abs().max().item() <= 64 * 2.0 ** -53 * b.abs().max().item()


@pytest.mark.parametrize("warped", [False, True])
@pytest.mark.parametrize("su,sp", [(0.0, 0.0), (0.0, 1.0), (1.0, 0.0), (2.0 ** -1000, 2.0 ** -1000), (2.0 ** 880, 2.0 ** 880),
                                   (2.0 ** -700, 1.0), (1.0, 2.0 ** -700), (2.0 ** 40, 2.0 ** -40)])
def test_scales(warped, su, sp):
    S, _ = _solver((3, 5, 4), warped, gamma_rho=1.0)
    rng = np.random.default_rng(7)
    x = rng.uniform(-1, 1, S.size())
    nu = S.sizes()[0]
    x[:nu] *= su
    x[nu:] *= sp
    t = torch.as_tensor(x, device="cuda")
    a, b = _both(S, lambda: S.vmult(t))
    for part in (slice(0, nu), slice(nu, None)):
        assert (a[part] - b[part]).abs().max().item() <= 64 * 2.0 ** -53 * b[part].abs().max().item()


@pytest.mark.parametrize("warped", [False, True])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf"), 1.7e308])
def test_values_out_of_range_spread_as_in_floating_point(warped, value):
    S, _ = _solver((5, 4, 3), warped, gamma_rho=1.0)
    rng = np.random.default_rng(9)
    x = torch.as_tensor(rng.uniform(-1, 1, S.size()), device="cuda")
    nu = S.sizes()[0]
    x[(3 * 9 + 4) * 11 + 5] = value      # a velocity node inside
    x[nu + 7] = value
    a, b = _both(S, lambda: S.vmult(x))
    assert torch.equal(torch.isfinite(a), torch.isfinite(b))
    ok = torch.isfinite(b)
    assert (a[ok] - b[ok]).abs().max().item() <= 64 * 2.0 ** -53 * b[ok].abs().max().item()
