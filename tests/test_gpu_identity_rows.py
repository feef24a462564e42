"""The identity rows of y = K x (16-byte packs with single entries at both ends): constrained rows return x bit for bit
and the rest is the operator, at every alignment of x and y, for row lengths around the packs."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("n,k,faces", [((1, 1), 2, 0xF), ((3, 2), 3, 0x5), ((1, 1, 1), 2, 0x3F), ((2, 1, 3), 2, 0x3D),
                                       ((3, 5, 2), 3, 0x21), ((2, 2, 1), 4, 0x3F)])
def test_every_alignment(n, k, faces, dtype):
    from paper_2205_15770_gb300 import StokesMG
    S = StokesMG(dim=len(n), n=n, n_levels=1, k=k, dirichlet_faces=faces, gamma_rho=1.0)
    m, nu = S.size(), S.sizes()[0]
    N = [k * v + 1 for v in n]
    g = np.meshgrid(*[np.arange(v) for v in N[::-1]], indexing="ij")[::-1]
    fixed = np.zeros(N[::-1], dtype=bool)
    for a in range(len(n)):
        fixed |= (bool(faces >> 2 * a & 1) & (g[a] == 0)) | (bool(faces >> 2 * a + 1 & 1) & (g[a] == N[a] - 1))
    rows = torch.as_tensor(np.concatenate([np.tile(fixed.reshape(-1), len(n)), np.zeros(m - nu, dtype=bool)]), device="cuda")
    x = torch.as_tensor(np.random.default_rng(1).uniform(-1, 1, m), dtype=dtype, device="cuda")
    ref = S.vmult(x)
    for ox in range(4):
        for oy in range(4):
            bx, by = torch.empty(m + 4, dtype=dtype, device="cuda"), torch.full((m + 8,), 7.0, dtype=dtype, device="cuda")
            bx[ox:ox + m] = x
            y = S.vmult(bx[ox:ox + m], by[oy:oy + m])
            assert torch.equal(y[rows], x[rows])
            eps = torch.finfo(dtype).eps  # atomics: another order of at most 8 summands
            assert (y - ref).abs().max() <= 16 * eps * ref.abs().max()
            assert (by[:oy] == 7.0).all() and (by[oy + m:] == 7.0).all()
