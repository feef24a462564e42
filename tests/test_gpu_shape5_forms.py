"""Launch shape 5 in FP32 (k = 2) has two kernels, the plane and the cell-component one: which of them runs is reported
(stokes_get_plane_form), a plain run's choice can be replayed (STOKES_TUNING's p32 list), and each of them, so chosen,
agrees with the FP64 operator and between its plain and fused smoothing."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu


def tuning(levels, plane=None, fused=0):
    j = lambda v: ",".join([str(v)] * levels)
    return f"s32={j(5)};s64={j(4)};f32={j(fused)};f64={j(0)}" + ("" if plane is None else f";p32={j(plane)}")


def mesh(n, warped, levels):
    return dict(dim=3, n=n, n_levels=levels, k=2, kA=1, kS=1, m=2, gamma_rho=5.0,
                vertices=W.perturbed_vertices(3, n, seed=1) if warped else None)


@pytest.mark.parametrize("n", [(1, 1, 1), (1, 1, 10), (7, 6, 5)])
@pytest.mark.parametrize("warped", [True, False])
def test_blocks_of_both_forms(n, warped, monkeypatch):
    from paper_2205_15770_gb300 import StokesMG
    S = {}
    for plane in (0, 1):
        monkeypatch.setenv("STOKES_TUNING", tuning(1, plane))
        S[plane] = StokesMG(dirichlet_faces=0x3F & ~0x8, **mesh(n, warped, 1))
        assert S[plane].launch_shapes(32) == [5] and S[plane].plane_levels(32) == [bool(plane)]
        assert S[plane].plane_levels(64) == [True]
    rng = np.random.default_rng(1)
    u, p = (torch.as_tensor(rng.uniform(-1, 1, m), dtype=torch.float32, device="cuda") for m in S[0].sizes())
    for blocks in (1, 2, 4, 3, 7):
        args = [u if blocks & 5 else None, p if blocks & 2 else None]
        ref = S[0].apply_blocks(blocks, *(a.double() if a is not None else None for a in args))
        both = [S[plane].apply_blocks(blocks, *args) for plane in (0, 1)]
        for y, z, r in zip(*both, ref):
            if r is not None:
                e = [(v.double() - r).norm().item() / r.norm().item() for v in (y, z)]
                # two FP32 evaluations of the same sums: the same size of error, or a few roundings
                assert max(e) <= max(2 * min(e), 8 * 2.0 ** -24), (blocks, e)


@pytest.mark.parametrize("n,warped", [((6, 10, 4), True), ((2, 4, 12), False)])
@pytest.mark.parametrize("plane", [0, 1])
def test_fused_smoothing_of_both_forms(n, warped, plane, monkeypatch):
    from paper_2205_15770_gb300 import StokesMG
    S = []
    for fused in (0, 1):
        monkeypatch.setenv("STOKES_TUNING", tuning(2, plane, fused))
        S.append(StokesMG(**mesh(n, warped, 2)))
        assert S[-1].fused_levels(32)[1] == bool(fused) and S[-1].plane_levels(32) == [bool(plane)] * 2
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    b, x = (torch.rand(S[0].size(), dtype=torch.float32, device="cuda", generator=g) * 2 - 1 for _ in range(2))
    for steps in (1, 3):
        a, r = (s.smooth(b, x.clone(), steps=steps) for s in S)
        assert (a - r).abs().max().item() <= 2e-4 * r.abs().max().item()  # ten times an FP32 operator's tolerance


def test_replay_of_a_plain_run(monkeypatch):
    import bench
    from paper_2205_15770_gb300 import StokesError, StokesMG
    kw = mesh((8, 8, 8), True, 3)
    S = StokesMG(**kw)
    choice = lambda s: [(s.launch_shapes(p), s.fused_levels(p), s.plane_levels(p)) for p in (32, 64)]
    monkeypatch.setenv("STOKES_TUNING", bench.tuning_string(S))
    assert choice(StokesMG(**kw)) == choice(S)
    monkeypatch.setenv("STOKES_NO_PLANE", "1")  # the cell-component form, as a run whose timing preferred it reports
    monkeypatch.setenv("STOKES_TUNING", tuning(3))
    C = StokesMG(**kw)
    assert C.plane_levels(32) == [False] * 3
    monkeypatch.delenv("STOKES_NO_PLANE")
    monkeypatch.setenv("STOKES_TUNING", bench.tuning_string(C))
    assert choice(StokesMG(**kw)) == choice(C)
    monkeypatch.setenv("STOKES_TUNING", tuning(3))  # without the list: the plane kernel where the level has it
    assert StokesMG(**kw).plane_levels(32) == [True] * 3
    monkeypatch.setenv("STOKES_TUNING", tuning(3, 1))
    with pytest.raises(StokesError):
        StokesMG(**{**kw, "k": 3, "vertices": None})
    monkeypatch.setenv("STOKES_TUNING", tuning(3, 2))
    with pytest.raises(StokesError):
        StokesMG(**kw)
