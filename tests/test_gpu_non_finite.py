"""An infinity or NaN among a smoother's inputs reaches no further through the explicit S~ (k = 2, k_A = 1) than through
its applications (STOKES_NO_SCHUR_MATRIX=1), and what stays finite stays the same: near a face, where the neighbours
along a row of nodes run into the next row."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fp32", [True, False])
@pytest.mark.parametrize("fuse", [True, False])
@pytest.mark.parametrize("n,at", [((32, 4), (31, 2)), ((32, 6, 4), (31, 3, 2)), ((6, 32, 4), (3, 31, 2)), ((4, 4, 32), (2, 2, 1))])
def test_reach_of_a_non_finite_pressure(n, at, fuse, fp32, monkeypatch):
    from paper_2205_15770_gb300 import StokesMG
    monkeypatch.setenv("STOKES_NO_AUTOTUNE", "1")
    if not fuse:
        monkeypatch.setenv("STOKES_NO_FUSE", "1")
    kw = dict(dim=len(n), n=n, n_levels=2, kA=1, kS=1, m=1, vcycle_fp32=fp32)
    S = StokesMG(**kw)
    monkeypatch.setenv("STOKES_NO_SCHUR_MATRIX", "1")
    C = StokesMG(**kw)
    dtype = torch.float32 if fp32 else torch.float64
    g = torch.Generator(device="cuda")
    g.manual_seed(1)
    b, x = (torch.rand(S.size(), dtype=dtype, device="cuda", generator=g) * 2 - 1 for _ in range(2))
    node = sum(v * int(torch.tensor([1] + [m + 1 for m in n[:a]]).prod()) for a, v in enumerate(at))
    for bad in (float("inf"), float("nan")):
        x[S.sizes()[0] + node] = bad
        before = S.launch_count
        y = S.smooth(b, x.clone())
        taken = S.launch_count - before
        before = C.launch_count
        z = C.smooth(b, x.clone())
        assert taken < C.launch_count - before
        fy, fz = y.isfinite(), z.isfinite()
        assert 0 < int(fz.sum()) < fz.numel()
        assert not bool((fz & ~fy).any()), int((fz & ~fy).sum())
        # two evaluations of the same sums of a few hundred terms
        assert (y[fz] - z[fz]).abs().max().item() <= 1e3 * torch.finfo(dtype).eps * z[fz].abs().max().item()
