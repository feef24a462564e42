"""The explicit matrix of a small level's FP32 cycle against the same cycle by launches (STOKES_NO_EXPLICIT=1) and the
FP64 cycle, for every kind of hierarchy that takes it: 2D and 3D, degrees, V and W, open outflow, per-cell viscosity."""
import numpy as np
import pytest
import torch

import workloads as W

pytestmark = pytest.mark.gpu

CASES = {
    "2d": dict(dim=2, n=(16, 16), n_levels=4),
    "2d warped, W-cycle, kA 3": dict(dim=2, n=(12, 20), n_levels=3, cycle="W", kA=3, kS=3, warped=True),
    "2d q3": dict(dim=2, n=(8, 8), n_levels=3, k=3),
    "2d q4": dict(dim=2, n=(8, 8), n_levels=3, k=4),
    "3d warped": dict(dim=3, n=(8, 8, 8), n_levels=3, warped=True, gamma_rho=100.0),
    "3d warped, W-cycle": dict(dim=3, n=(8, 8, 8), n_levels=3, warped=True, cycle="W"),
    "3d channel": dict(dim=3, n=(12, 8, 8), n_levels=3, hi=(4.0, 1.0, 1.0), dirichlet_faces=0x3F & ~0x2, mu=1e-3),
    "3d per-cell viscosity": dict(dim=3, n=(8, 8, 8), n_levels=3, cells=True),
    "3d symmetric gradient": dict(dim=3, n=(8, 8, 8), n_levels=3, sym_grad=True),
}


@pytest.mark.parametrize("name", list(CASES))
def test_explicit_level_is_the_cycle(name, monkeypatch):
    from paper_2205_15770_gb300 import StokesMG
    kw = dict(CASES[name])
    if kw.pop("warped", False):
        kw["vertices"] = W.perturbed_vertices(kw["dim"], kw["n"], seed=2)
    if kw.pop("cells", False):
        kw["mu_cell"] = np.exp(np.random.default_rng(1).standard_normal(int(np.prod(kw["n"]))))
    kw = {**dict(kA=1, kS=1, m=2), **kw}

    def cycles():
        S = StokesMG(**kw)
        rng = np.random.default_rng(4)
        out = []
        for _ in range(2):  # a second right-hand side on the same buffers
            b = torch.as_tensor(rng.uniform(-1, 1, S.size()), device="cuda")
            nu = S.sizes()[0]
            b[:nu] = S.mass(b[:nu].contiguous(), full_rows=False)  # zero on Dirichlet nodes
            b[nu:] -= b[nu:].mean()
            b = b.float()
            before = S.launch_count
            x32 = S.vcycle(b)
            out.append((x32.double(), S.vcycle(b.double()), S.launch_count - before))
        return out

    explicit = cycles()
    monkeypatch.setenv("STOKES_NO_EXPLICIT", "1")
    launches = cycles()
    assert explicit[1][2] < launches[1][2]
    for (xe, x64, _), (xl, _, _) in zip(explicit, launches):
        ee, el = ((x - x64).norm().item() / x64.norm().item() for x in (xe, xl))
        # both are FP32 evaluations of the same map, 1e-7 to 1e-6 off the FP64 cycle: within a factor of two of
        # each other, or below 8 roundings
        assert ee <= max(2 * el, 8 * 2.0 ** -24), (ee, el)
