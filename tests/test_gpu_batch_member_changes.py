"""A batch whose member's viscosities or launch shape change after a batched solve or cycle: the next one is captured again from
the members as they are then (a change of viscosities replaces the member's vectors)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["graphs", "queue", "host"])
def test_solve_after_a_change(mode, monkeypatch):
    from paper_2205_15770_gb300 import StokesBatch, StokesMG
    if mode != "graphs":
        monkeypatch.setenv({"queue": "STOKES_BATCH_QUEUE", "host": "STOKES_HOST_KRYLOV"}[mode], "1")
    rng = np.random.default_rng(0)
    kw = dict(kA=1, kS=1, m=2, schur_diag="d")
    Bt = StokesBatch([dict(dim=3, n=(4, 4, 4), n_levels=2, gamma_rho=1.0), dict(dim=3, n=(8, 8, 8), n_levels=3)], **kw)
    bs = [mv.mass_rhs(torch.as_tensor(rng.uniform(-1, 1, mv.sizes()[0]), device="cuda")) for mv in Bt.members]
    mu = np.exp(rng.standard_normal(512))

    def check():
        xs, its, _ = Bt.solve(bs, rtol=1e-8)
        for b, mv, x in zip(bs, Bt.members, xs):
            assert torch.linalg.norm(b - mv.vmult(x)).item() <= 1.01e-8 * torch.linalg.norm(b).item()
        return its

    check()
    if mode == "queue":
        Bt.vcycle([b.float() for b in bs])
    Bt.members[1].set_viscosity(mu)
    its = check()
    assert Bt.krylov_mode == {"graphs": 1, "queue": 2, "host": 0}[mode]
    S = StokesMG(3, (8, 8, 8), 3, mu_cell=mu, **kw)
    assert abs(its[1] - S.solve(bs[1], rtol=1e-8)[1]) <= 1
    if mode == "queue":
        x = Bt.vcycle([b.float() for b in bs])[1].double()
        ref = S.vcycle(bs[1])
        own = S.vcycle(bs[1].float()).double()
        # as accurate as the member's own FP32 cycle, or 1e-5 (the bound of the queue's cycles elsewhere)
        assert (x - ref).abs().max() <= max(2 * (own - ref).abs().max().item(), 1e-5 * ref.abs().max().item())
    Bt.members[1].set_launch_shape(2, 4, 32)
    check()
    Bt.close()
