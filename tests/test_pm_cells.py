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


def test_meshes_beyond_32_bit_batches():
    """N = 896, the first mesh whose three component meshes pass 2^31 values, against the same method
    in FP64 by torch on the GPU.  2000 particles in a few clumps, so that the field is not noise."""
    N, L = 896, 7.0
    r_s, d = 1.2 * L / N, L / N
    rng = np.random.default_rng(0)
    pos = np.mod(np.repeat(rng.random((40, 3)) * L, 50, 0) + 3 * d * rng.standard_normal((2000, 3)), L)
    mass = rng.uniform(0.5, 1.5, 2000)
    p, m = torch.tensor(pos, device="cuda"), torch.tensor(mass, device="cuda")
    got = psr.PM(N).forces(p, m, L, r_s).double()
    u = p * (N / L)
    i0 = u.floor().long().clamp(max=N - 1)
    f = u - i0
    rho = torch.zeros(N ** 3, dtype=torch.float64, device="cuda")
    corners = []
    for a in range(8):
        b = [(a >> q) & 1 for q in range(3)]
        ix, iy, iz = ((i0[:, q] + b[q]) % N for q in range(3))
        w = torch.ones_like(m)
        for q in range(3):
            w = w * (f[:, q] if b[q] else 1.0 - f[:, q])
        corners.append(((ix * N + iy) * N + iz, w))
        rho.index_add_(0, corners[-1][0], w * m)
    k1 = 2 * np.pi / L * torch.fft.fftfreq(N, 1.0 / N, dtype=torch.float64, device="cuda")
    kz = 2 * np.pi / L * torch.arange(N // 2 + 1, dtype=torch.float64, device="cuda")
    ks = [k1[:, None, None], k1[None, :, None], kz[None, None, :]]
    phi = torch.fft.rfftn(rho.reshape(N, N, N) / d ** 3)
    del rho
    k2 = ks[0] ** 2 + ks[1] ** 2 + ks[2] ** 2
    k2[0, 0, 0] = 1.0
    phi *= -4 * np.pi * torch.exp(-k2 * r_s ** 2) / k2
    del k2
    for k in ks:
        phi /= torch.sinc(k * (0.5 * d / np.pi)) ** 4
    phi[0, 0, 0] = 0.0
    ref = torch.zeros_like(p)
    for q, k in enumerate(ks):
        k = k.clone()
        k.view(-1)[N // 2] = 0.0
        g = torch.fft.irfftn(-1j * k * phi, s=(N, N, N)).reshape(-1)
        for at, w in corners:
            ref[:, q] += w * g[at]
        del g
    assert float(((got - ref).square().sum() / ref.square().sum()).sqrt()) < 2e-5
