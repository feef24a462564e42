"""The FP32 plane kernel (launch shape 5, k = 2) against the FP64 operator and the cell-component kernel
(STOKES_NO_PLANE=1), block by block at the edges of its groups of ten cells, and its fused smoothing."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(1, 1, 1), (1, 1, 10), (3, 5, 7), (11, 2, 1), (7, 6, 5)])
@pytest.mark.parametrize("warped,cells", [(True, False), (False, False), (False, True), (True, True)])
def test_blocks(n, warped, cells, monkeypatch):
    from paper_2205_15770_gb300 import StokesMG
    rng = np.random.default_rng(1)
    kw = dict(dim=3, n=n, n_levels=1, k=2, gamma_rho=5.0, dirichlet_faces=0x3F & ~0x8, hi=(1.0, 2.0, 0.5) if not warped else (1.0,) * 3,
              vertices=W.perturbed_vertices(3, n, seed=1) if warped else None,
              mu_cell=rng.uniform(0.2, 5.0, int(np.prod(n))) if cells else None)
    S = StokesMG(**kw)
    monkeypatch.setenv("STOKES_NO_PLANE", "1")
    C = StokesMG(**kw)
    for s in (S, C):
        s.set_launch_shape(0, 5, 32)
    S.set_launch_shape(0, 4, 64)
    nu, npr = S.sizes()
    u, p = (torch.as_tensor(rng.uniform(-1, 1, m), dtype=torch.float32, device="cuda") for m in (nu, npr))
    for blocks in (1, 2, 4, 3, 7):
        args = [blocks, u if blocks & 5 else None, p if blocks & 2 else None]
        ref = S.apply_blocks(blocks, *(a.double() if a is not None else None for a in args[1:]))
        for y, z, r in zip(S.apply_blocks(*args), C.apply_blocks(*args), ref):
            if r is not None:
                e, c = ((v.double() - r).norm().item() / r.norm().item() for v in (y, z))
                # two FP32 evaluations of the same sums: the same size of error, or a few roundings
                assert e <= max(2 * c, 8 * 2.0 ** -24), (blocks, e, c)


@pytest.mark.parametrize("n,warped", [((6, 10, 4), True), ((2, 4, 12), False)])
@pytest.mark.parametrize("kS", [1, 2])
def test_fused_smoothing(n, warped, kS, monkeypatch):
    from paper_2205_15770_gb300 import StokesMG
    monkeypatch.setenv("STOKES_NO_AUTOTUNE", "1")
    kw = dict(dim=3, n=n, n_levels=2, k=2, kA=1, kS=kS, m=2, gamma_rho=1.0,
              vertices=W.perturbed_vertices(3, n, seed=3) if warped else None)
    F = StokesMG(**kw)
    monkeypatch.setenv("STOKES_NO_FUSE", "1")
    U = StokesMG(**kw)
    for s in (F, U):
        s.set_launch_shape(1, 5, 32)
    assert F.fused_levels(32)[1] and not U.fused_levels(32)[1]
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    b, x = (torch.rand(F.size(), dtype=torch.float32, device="cuda", generator=g) * 2 - 1 for _ in range(2))
    for steps in (1, 3):
        a, r = F.smooth(b, x.clone(), steps=steps), U.smooth(b, x.clone(), steps=steps)
        assert (a - r).abs().max().item() <= 2e-4 * r.abs().max().item()  # ten times an FP32 operator's tolerance
