"""A member's own cycle and the batch's work-queue cycle run on the same work vectors, the queue always in the unfused
smoother form, the member's own where it is faster in the fused one, which starts from vectors that are zero: after a queue
cycle (of another, larger right-hand side) the member's own cycle is what it was before."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kS", [1, 2])
@pytest.mark.parametrize("solve", [False, True])
def test_member_cycle_after_the_queue(solve, kS, monkeypatch):
    from paper_2205_15770_gb300 import StokesBatch
    monkeypatch.setenv("STOKES_NO_AUTOTUNE", "1")
    monkeypatch.setenv("STOKES_BATCH_QUEUE", "1")
    Bt = StokesBatch([dict(dim=3, n=(4, 4, 4), n_levels=2, gamma_rho=1.0), dict(dim=3, n=(8, 8, 8), n_levels=3)], kA=1, kS=kS,
                     m=1, schur_diag="d")
    assert all(mv.fused_levels(32)[-1] for mv in Bt.members)
    rng = np.random.default_rng(0)
    bs = [mv.mass_rhs(torch.as_tensor(rng.uniform(-1, 1, mv.sizes()[0]), device="cuda")) for mv in Bt.members]
    refs = [mv.vcycle(b) for mv, b in zip(Bt.members, bs)]
    before = [mv.vcycle(b.float()).double() for mv, b in zip(Bt.members, bs)]
    if solve:
        Bt.solve(bs, rtol=1e-8)
        assert Bt.krylov_mode == 2
    else:
        Bt.vcycle([1e4 * b.float() for b in bs])
    for mv, b, ref, x in zip(Bt.members, bs, refs, before):
        after = mv.vcycle(b.float()).double()
        e0, e1 = ((v - ref).norm().item() / ref.norm().item() for v in (x, after))
        # FP32 evaluations of one map: within a factor of two of each other, or below 8 roundings
        assert e1 <= max(2 * e0, 8 * 2.0 ** -24), (e1, e0)
    Bt.close()
