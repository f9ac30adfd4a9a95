"""The PM deposit's two meshes (pairs of cells that start at an even and at an odd z) and the
interpolation's float4 mesh, at every parity and wrap of the cells, on the smallest meshes.

Tolerance: 2e-5 relative RMS against the FP64 mesh method, the bound of the PM tests."""
import numpy as np
import pytest
import torch

import paper_2107_14008_gb300 as psr
from oracle import pm as opm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_pm", [8, 10, 12, 22])
@pytest.mark.parametrize("deconvolve", [True, False])
def test_every_cell_parity_and_wrap(n_pm, deconvolve):
    L = 5.0
    d = L / n_pm
    rng = np.random.default_rng(n_pm)
    edge = np.array([0.0, 0.5 * d, d, L - d, L - 1e-9, np.nextafter(L, 0.0), L, -1e-300, -0.0, -0.3 * d, 7 * L + 0.2])
    grid = np.stack(np.meshgrid(edge, edge[::3], edge, indexing="ij"), -1).reshape(-1, 3)
    pos = np.concatenate([grid, rng.random((500, 3)) * L, rng.integers(0, n_pm, (200, 3)) * d])
    mass = rng.uniform(0.5, 1.5, len(pos))
    r_s = 1.2 * d
    ref = opm.pm_forces(pos, mass, L, r_s, n_pm, deconvolve=deconvolve)
    p, m = torch.tensor(pos, device="cuda"), torch.tensor(mass, device="cuda")
    pm = psr.PM(n_pm)
    got = pm.forces(p, m, L, r_s, deconvolve=deconvolve)
    g = got.double().cpu().numpy()
    assert np.sqrt(((g - ref) ** 2).sum() / (ref ** 2).sum()) < 2e-5
    base = torch.full_like(got, 3.0)
    bad = p.clone()
    bad[5, 1], bad[17, 2] = float("nan"), float("inf")
    out = pm.forces(bad, m, L, r_s, out=base, accumulate=True, deconvolve=deconvolve)
    assert torch.all(out[[5, 17]] == 3.0) and torch.isfinite(out).all()
