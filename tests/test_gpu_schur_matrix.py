"""The explicit S~ of the smoother (k = 2, k_A = 1) against S~ by its applications (STOKES_NO_SCHUR_MATRIX=1) and the
FP64 smoother, in both precisions and smoother forms: grids smaller than the stencil, rows that end inside a block of
32, several and partial batches of probes, open boundaries, density and viscosity per cell, symmetric gradient."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

CASES = {
    "2d, 3 x 5 nodes": dict(dim=2, n=(2, 4), n_levels=2),
    "2d warped, kS 4": dict(dim=2, n=(24, 10), n_levels=2, kS=4, warped=True),
    "3d, 3 nodes": dict(dim=3, n=(2, 2, 2), n_levels=2),
    "3d box, kS 2": dict(dim=3, n=(4, 10, 6), n_levels=2, kS=2, gamma_rho=50.0),
    "3d warped channel": dict(dim=3, n=(12, 8, 8), n_levels=3, warped=True, dirichlet_faces=0x3F & ~0x2),
    "3d symmetric gradient, kS 3": dict(dim=3, n=(6, 4, 8), n_levels=2, sym_grad=True, kS=3),
    "3d per cell": dict(dim=3, n=(4, 4, 12), n_levels=2, cells=True, gamma_rho=10.0),
}


@pytest.mark.parametrize("fp32", [True, False])
@pytest.mark.parametrize("fuse", [True, False])
@pytest.mark.parametrize("name", list(CASES))
def test_smoothing_with_the_explicit_schur_complement(name, fuse, fp32, monkeypatch):
    from paper_2205_15770_gb300 import StokesMG
    kw = dict(CASES[name])
    nc = int(np.prod(kw["n"]))
    if kw.pop("warped", False):
        kw["vertices"] = W.perturbed_vertices(kw["dim"], kw["n"], seed=2)
    if kw.pop("cells", False):
        rng = np.random.default_rng(1)
        kw["mu_cell"] = np.exp(rng.standard_normal(nc))
        kw["rho_cell"] = np.exp(rng.standard_normal(nc))
    kw = {**dict(kA=1, kS=1, m=2, vcycle_fp32=fp32), **kw}
    monkeypatch.setenv("STOKES_NO_AUTOTUNE", "1")
    if not fuse:
        monkeypatch.setenv("STOKES_NO_FUSE", "1")
    dtype = torch.float32 if fp32 else torch.float64

    def smoothed():
        S = StokesMG(**kw)
        rng = np.random.default_rng(4)
        out = []
        for _ in range(2):  # a second right-hand side on the same buffers
            b, x = (torch.as_tensor(rng.uniform(-1, 1, S.size()), dtype=dtype, device="cuda") for _ in range(2))
            before = S.launch_count
            out.append((S.smooth(b, x.clone(), steps=2).double(), S.launch_count - before, b, x))
        return out, S

    matrix, _ = smoothed()
    monkeypatch.setenv("STOKES_NO_SCHUR_MATRIX", "1")
    chain, S = smoothed()
    for (xm, nm, b, x), (xc, ncn, _, _) in zip(matrix, chain):
        assert nm < ncn
        x64 = S.smooth(b.double(), x.double(), steps=2)
        em, ec = ((v - x64).norm().item() / x64.norm().item() for v in (xm, xc))
        # two evaluations of the same map: within a factor of two of each other, or below 16 roundings
        eps = 2.0 ** -24 if fp32 else 2.0 ** -53
        assert em <= max(2 * ec, 16 * eps), (em, ec)
