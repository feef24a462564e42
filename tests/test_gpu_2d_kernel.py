"""The 2D cell kernel (a thread per cell and component) against the point kernel (launch shape -1), block by block, at
cell counts around its warps of 32 cells, and its fused smoothing against the unfused one."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu
# two sums of the same terms in another order: k = 4 has 25 terms a sweep and direction
TOL = {torch.float64: 1e-13, torch.float32: 2e-5}


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("k", [2, 3, 4])
@pytest.mark.parametrize("n,warped,faces", [((1, 1), False, 0xF), ((31, 1), True, 0xF), ((3, 11), False, 0xD), ((5, 13), True, 0x5)])
def test_blocks_match_the_point_kernel(n, warped, faces, k, dtype):
    from paper_2205_15770_gb300 import StokesMG
    rng = np.random.default_rng(1)
    if k == 4 and n == (31, 1):
        n = (7, 1)
    S = StokesMG(dim=2, n=n, n_levels=1, k=k, dirichlet_faces=faces, gamma_rho=3.0,
                 vertices=W.perturbed_vertices(2, n, seed=1) if warped else None,
                 mu_cell=rng.uniform(0.5, 2.0, n[0] * n[1]))
    nu, npr = S.sizes()
    u, p = (torch.as_tensor(rng.uniform(-1, 1, m), dtype=dtype, device="cuda") for m in (nu, npr))
    prec = 64 if dtype == torch.float64 else 32
    for blocks in (1, 2, 4, 3, 7):
        out = []
        for shape in (4, -1):
            S.set_launch_shape(0, shape, prec)
            out.append(S.apply_blocks(blocks, u=u if blocks & 5 else None, p=p if blocks & 2 else None))
        for a, b in zip(*out):
            if a is not None:
                assert (a - b).abs().max().item() <= TOL[dtype] * b.abs().max().item(), blocks


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("kS", [1, 3])
@pytest.mark.parametrize("n,k,warped", [((6, 10), 2, True), ((34, 2), 2, False), ((4, 6), 3, True)])
def test_fused_smoothing_matches_the_unfused(n, k, warped, kS, dtype, monkeypatch):
    from paper_2205_15770_gb300 import StokesMG
    monkeypatch.setenv("STOKES_NO_AUTOTUNE", "1")  # the fused form wherever it is eligible
    kw = dict(dim=2, n=n, n_levels=2, k=k, kA=1, kS=kS, m=2, gamma_rho=1.0,
              vertices=W.perturbed_vertices(2, n, seed=3) if warped else None)
    F = StokesMG(**kw)
    monkeypatch.setenv("STOKES_NO_FUSE", "1")
    U = StokesMG(**kw)
    prec = 64 if dtype == torch.float64 else 32
    assert F.fused_levels(prec)[1] and not U.fused_levels(prec)[1]
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    b, x = (torch.rand(F.size(), dtype=dtype, device="cuda", generator=g) * 2 - 1 for _ in range(2))
    for steps in (1, 3):
        a, r = F.smooth(b, x.clone(), steps=steps), U.smooth(b, x.clone(), steps=steps)
        assert (a - r).abs().max().item() <= 10 * TOL[dtype] * r.abs().max().item()
    z, y = F.vcycle(b), U.vcycle(b)
    assert (z - y).abs().max().item() <= 100 * TOL[dtype] * y.abs().max().item()
