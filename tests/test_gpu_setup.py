"""What the setup computes in batched launches, against dense linear algebra on the same operator: the coarse inverse
(one launch a Gauss-Jordan step up to 1,024 rows, two above), the probed Schur diagonal "d" (several colours a launch)
and the largest eigenvalue from Lanczos with its coefficients on the device (also where it runs out of dimensions)."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [
    dict(dim=3, n=(4, 4, 4), n_levels=2, warped=True),
    dict(dim=3, n=(4, 4, 4), n_levels=2, sym_grad=True, mu=0.5),
    dict(dim=3, n=(4, 4, 4), n_levels=2, gamma_rho=3.0, dirichlet_faces=0x3D),
    dict(dim=3, n=(4, 4, 4), n_levels=2, c_mass=0.1),
    dict(dim=3, n=(6, 6, 8), n_levels=2),  # 1,029 + 80 + 1 rows
])
def test_coarse_inverse(kw):
    from paper_2205_15770_gb300 import StokesMG
    kw = dict(kw)
    if kw.pop("warped", False):
        kw["vertices"] = W.perturbed_vertices(kw["dim"], kw["n"], seed=1)
    S = StokesMG(kA=1, kS=1, **kw)
    x = torch.as_tensor(np.random.default_rng(0).uniform(-1, 1, S.size(0)), device="cuda")
    b = S.vmult(x, level=0)
    r = S.vmult(S.coarse_solve(b), level=0) - b
    # rows x 2^-52 x condition number (below 1e4 on these meshes of one to four cells a direction)
    assert r.norm().item() <= S.size(0) * 2.0 ** -52 * 1e4 * b.norm().item()


def columns(S, blocks, level, n):
    e = torch.zeros(n, dtype=torch.float64, device="cuda")
    out = []
    for j in range(n):
        e[j] = 1.0
        yu, yp = S.apply_blocks(blocks, u=e, level=level)
        out.append((yu if yu is not None else yp).clone())
        e[j] = 0.0
    return torch.stack(out, dim=1)


@pytest.mark.parametrize("restart", [30, 1])
@pytest.mark.parametrize("warped", [False, True])
def test_schur_diagonal_d(warped, restart):
    from paper_2205_15770_gb300 import StokesMG
    n = (4, 6, 2)
    v = W.perturbed_vertices(3, n, seed=3) if warped else None
    S = StokesMG(3, n, 2, vertices=v, kA=1, kS=1, schur_diag="d", restart=restart)
    DA, DS = S.diagonals(1)
    B = columns(S, 4, 1, S.sizes(1)[0])
    ref = (B * B / DA).sum(dim=1)
    assert ((DS - ref).abs() / ref).max().item() <= 1e-12  # sums of at most 375 terms, each a few roundings


@pytest.mark.parametrize("dim,n", [(2, (2, 2)), (3, (2, 2, 2))])
def test_lanczos_beyond_the_dimension(dim, n):
    from paper_2205_15770_gb300 import StokesMG
    S = StokesMG(dim, n, 2, kA=1, kS=1, eig_iters=120, eig_safety=1.0)
    DA, _ = S.diagonals(1)
    A = columns(S, 1, 1, S.sizes(1)[0])
    s = DA.rsqrt()
    lam = torch.linalg.eigvalsh((s[:, None] * A * s).cpu()).max().item()
    # an extreme Ritz value, its error the square of the residual's: far below the tolerance after all the dimensions
    assert abs(S.level_params(1)["beta_A"] - lam) <= 1e-8 * lam


@pytest.mark.parametrize("fp32", [True, False])
def test_change_of_viscosities_keeps_the_tuned_choices(fp32):
    from paper_2205_15770_gb300 import StokesMG
    n, rng = (8, 8, 8), np.random.default_rng(5)
    mu = [np.exp(rng.standard_normal(512)) for _ in range(3)]
    kw = dict(vertices=W.perturbed_vertices(3, n, seed=1), kA=1, kS=1, vcycle_fp32=fp32)
    S = StokesMG(3, n, 3, mu_cell=mu[0], **kw)
    tuned = [(S.launch_shapes(p), S.fused_levels(p), S.geometry_stored(p)) for p in (32, 64)]
    S.set_launch_shape(2, 1, 64)  # a caller's shape lasts until the next change of viscosities
    for m in mu[1:]:
        S.set_viscosity(m)
        assert [(S.launch_shapes(p), S.fused_levels(p), S.geometry_stored(p)) for p in (32, 64)] == tuned
        F = StokesMG(3, n, 3, mu_cell=m, **kw)
        x = torch.as_tensor(rng.uniform(-1, 1, S.size()), device="cuda")
        ref = F.vcycle(x)
        # FP64 evaluations of one map by kernels that may differ: a few hundred roundings
        assert (S.vcycle(x) - ref).norm().item() <= 1e-13 * ref.norm().item()
