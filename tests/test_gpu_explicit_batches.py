"""The explicit matrix of a small level where its columns are built in batches of 512 and the last batch is a single one
(1,025 unknowns): that column, like the others, is the cycle by launches.  The viscosity jumps, so that what a former batch
left in the work vectors is not small against the last column."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,kS", [(1, 1), (1, 2), (2, 1)])
@pytest.mark.parametrize("fused", [True, False])
def test_single_last_column(fused, m, kS, monkeypatch):
    from paper_2205_15770_gb300 import StokesMG
    n = (4, 88)
    mu = np.ones((n[1], n[0]))
    mu[:n[1] // 2] = 1e-2
    kw = dict(dim=2, n=n, n_levels=3, kA=1, kS=kS, m=m, hi=(1.0, 22.0), mu_cell=mu.reshape(-1))
    monkeypatch.setenv("STOKES_NO_AUTOTUNE", "1")
    if not fused:
        monkeypatch.setenv("STOKES_NO_FUSE", "1")
    E = StokesMG(**kw)
    assert E.size(1) == 1025 and E.fused_levels(32)[1] == fused
    monkeypatch.setenv("STOKES_NO_EXPLICIT", "1")
    L = StokesMG(**kw)
    # the right-hand side's last entries are those that the last column multiplies
    b = torch.zeros(E.size(), device="cuda")
    b[-3:] = torch.as_tensor(np.random.default_rng(3).uniform(1, 2, 3), device="cuda")
    ref = L.vcycle(b.double())
    ee, el = ((S.vcycle(b).double() - ref).norm().item() / ref.norm().item() for S in (E, L))
    # FP32 evaluations of one map: within a factor of two of each other, or below 8 roundings
    assert ee <= max(2 * el, 8 * 2.0 ** -24), (ee, el)
