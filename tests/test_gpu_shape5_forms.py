"""Launch shape 5 in FP32 (k = 2) has two kernels, the plane and the cell-component one: which of them runs is reported
(stokes_get_plane_form) and a plain run's choice can be replayed (STOKES_TUNING's p32 list)."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def tuning(levels, plane=None, fused=0):
    j = lambda v: ",".join([str(v)] * levels)
    return f"s32={j(5)};s64={j(4)};f32={j(fused)};f64={j(0)}" + ("" if plane is None else f";p32={j(plane)}")


def mesh(n, warped, levels):
    return dict(dim=3, n=n, n_levels=levels, k=2, kA=1, kS=1, m=2, gamma_rho=5.0,
                vertices=W.perturbed_vertices(3, n, seed=1) if warped else None)


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
