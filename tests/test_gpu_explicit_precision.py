"""The explicit matrix of a small level keeps the precision of the launches it replaces, whose coarse solve sums in FP64:
the FP32 cycle without smoothing steps (restriction, coarse solve, prolongation; no atomics, so the same on every run)
is on average over sixteen right-hand sides no further from the FP64 cycle than by launches (STOKES_NO_EXPLICIT=1).  With
smoothing, the columns of a 2D matrix come from the 2D kernel (from the point kernel they left 1.12 to 1.19 times the error)."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

CASES = {
    "2d": dict(dim=2, n=(24, 40), n_levels=3),
    "2d, four levels": dict(dim=2, n=(32, 32), n_levels=4, vertices=W.perturbed_vertices(2, (32, 32), seed=2)),
    "2d q3": dict(dim=2, n=(16, 16), n_levels=4, k=3),
    "3d warped": dict(dim=3, n=(8, 8, 8), n_levels=3, vertices=W.perturbed_vertices(3, (8, 8, 8), seed=2)),
    "3d channel": dict(dim=3, n=(12, 8, 8), n_levels=3, hi=(4.0, 1.0, 1.0), dirichlet_faces=0x3F & ~0x2, mu=1e-3),
    "3d density": dict(dim=3, n=(8, 8, 8), n_levels=3, gamma_rho=1e4),
    "2d warped, smoothing": dict(dim=2, n=(24, 40), n_levels=4, m=2, gamma_rho=100.0, schur_diag="d",
                                 vertices=W.perturbed_vertices(2, (24, 40), seed=1)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_error_of_the_coarse_solve(name, monkeypatch):
    from paper_2205_15770_gb300 import StokesMG
    kw = {**dict(kA=1, kS=1, m=0), **CASES[name]}
    E = StokesMG(**kw)
    monkeypatch.setenv("STOKES_NO_EXPLICIT", "1")
    L = StokesMG(**kw)
    nu, err = E.sizes()[0], []
    for seed in range(16):
        b = torch.as_tensor(np.random.default_rng(seed).uniform(-1, 1, E.size()), device="cuda")
        b[:nu] = E.mass(b[:nu].contiguous(), full_rows=False)  # zero on Dirichlet nodes
        b[nu:] -= b[nu:].mean()
        b = b.float()
        ref = L.vcycle(b.double())
        err.append([((S.vcycle(b).double() - ref).norm() / ref.norm()).item() for S in (E, L)])
    explicit, launches = np.exp(np.log(err).mean(axis=0))
    # with smoothing the atomics' order moves the mean of sixteen by up to 3 %
    assert explicit <= (1.05 if kw["m"] else 1.0) * launches, (explicit, launches)
