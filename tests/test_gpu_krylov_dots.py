"""The device Krylov loop's grouped dot products (eight vectors a pass) and its update with the norm, against the
host-driven loop (STOKES_HOST_KRYLOV=1: a vector at a time): restart lengths around a group, several groups, sizes that
are no multiple of a block."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("restart", [7, 8, 9, 20])
@pytest.mark.parametrize("dim,n", [(2, (6, 10)), (3, (4, 4, 6))])
def test_device_loop_matches_the_host_loop(dim, n, restart, monkeypatch):
    from paper_2205_15770_gb300 import StokesError, StokesMG
    rng = np.random.default_rng(3)
    kw = dict(kA=1, kS=1, m=1, restart=restart, vcycle_fp32=False, mu_cell=np.exp(2 * rng.standard_normal(int(np.prod(n)))))
    f = rng.uniform(-1, 1, 10 ** 5)
    out = []
    for host in (False, True):
        if host:
            monkeypatch.setenv("STOKES_HOST_KRYLOV", "1")
        S = StokesMG(dim, n, 2, **kw)
        b = S.mass_rhs(torch.as_tensor(f[:S.sizes()[0]], device="cuda"))
        x = torch.zeros_like(b)
        with pytest.raises(StokesError, match="maxit"):  # 20 steps, unconverged: x holds the last iterate
            S.solve(b, x=x, rtol=1e-14, maxit=20)
        assert S.krylov_mode == (0 if host else 1)
        out.append(x)
    # the same iterates up to the rounding that 20 steps amplify
    assert (out[0] - out[1]).norm().item() <= 1e-6 * out[1].norm().item()
