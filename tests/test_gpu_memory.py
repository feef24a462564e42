"""Device memory of a setup: optional tables never cost a setup that fits without them, and work space is given back."""
import gc

import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

MB = 1 << 20


def free_memory():
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_setup_without_room_for_the_plane_tables(monkeypatch):
    """A warped 24^3 mesh with room for the context but not for the plane kernels' coefficients: by their own test (a
    quarter of the free memory) they fit, the vectors allocated after them then do not."""
    from paper_2205_15770_gb300 import StokesMG
    n = (24, 24, 24)
    cells = 24 ** 3 * 9 // 8
    table = 3694 * cells  # FP64; FP32: 2304 * cells more
    kw = dict(dim=3, n=n, n_levels=4, vertices=W.perturbed_vertices(3, n, seed=1), kA=1, kS=1, restart=60)
    S = StokesMG(**kw)  # every kernel is loaded from here on
    f = torch.as_tensor(W.fourier_forcing(3, 2, n, seed=1).reshape(-1), device="cuda")
    b = S.mass_rhs(f)
    ref, its, _ = S.solve(b, rtol=1e-8)
    S.close()
    del S
    for name in ("STOKES_NO_PLANE", "STOKES_NO_SCHUR_MATRIX", "STOKES_NO_EXPLICIT"):
        monkeypatch.setenv(name, "1")
    before = free_memory()
    S = StokesMG(**kw)
    need = before - free_memory() - table
    S.close()
    del S
    for name in ("STOKES_NO_PLANE", "STOKES_NO_SCHUR_MATRIX", "STOKES_NO_EXPLICIT"):
        monkeypatch.delenv(name)
    left = need + 48 * MB
    assert need > 4 * table > 4 * 48 * MB  # the tables pass their own test and do not fit beside the rest
    hog = []
    try:
        while (free := free_memory()) > left + 2 * MB:
            hog.append(torch.empty(min(free - left, 32 << 30), dtype=torch.uint8, device="cuda"))
        S = StokesMG(**kw)
        x, its2, rel = S.solve(b, rtol=1e-8)
        assert its2 <= its + 1 and (x - ref).norm().item() <= 1e-5 * ref.norm().item()
        S.close()
    finally:
        hog.clear()
        free_memory()



def test_coarse_factorisation_keeps_only_the_inverse():
    """5^3 cells on the coarsest level: 4,210 rows, an inverse of 142 MB beside 60 MB of vectors; the matrix (142 MB) and the
    augmented one (284 MB) are work of the setup."""
    from paper_2205_15770_gb300 import StokesMG
    kw = dict(dim=3, n=(10, 10, 10), n_levels=2, kA=1, kS=1)
    StokesMG(3, (2, 2, 2), 1).close()  # the library and the static scratch are loaded
    before = free_memory()
    S = StokesMG(**kw)
    assert before - free_memory() <= (142 + 2 * 60) * MB
    S.close()
