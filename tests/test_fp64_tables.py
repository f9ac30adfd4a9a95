"""The FP64 kernels' T and exp(-x^2) tables, cull, lane filling and shared rows, over cutoffs from
x_c = 0.3 to beyond the tables' end (x = 12), leaf sizes and both mass forms.

Tolerance: every factor of a pair is exact to a few FP64 roundings (2^-53 each, the tables' left-out
term below 1e-16), and a target sums some hundred terms: 1e-13 relative RMS (a wrong node,
coefficient, image or target is orders above that)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2107_14008_gb300 as psr

pytestmark = pytest.mark.gpu


def _rms(a, b):
    return float(np.sqrt(((a - b) ** 2).sum() / (b ** 2).sum()))


@pytest.mark.parametrize("x_c", [0.3, 2.25, 5.99, 6.01, 9.0, 14.0])
@pytest.mark.parametrize("max_leaf,n", [(1, 90), (7, 700), (32, 1500), (64, 1500)])
@pytest.mark.parametrize("equal", [True, False])
def test_fp64_matches_oracle(x_c, max_leaf, n, equal):
    rng = np.random.default_rng(5)
    L, r_c = 30.0, 13.0
    r_s = r_c / (2.0 * x_c)
    pos = rng.random((n, 3)) * L
    pos[: n // 4] = 29.0 + 1.5 * rng.standard_normal((n // 4, 3))  # a clump across the box's corner
    pos = np.mod(pos, L)
    pos[n // 2] = pos[n // 2 + 1]  # a coincident pair
    mass = np.full(n, 1.0 / n) if equal else rng.uniform(0.2, 2.0, n) / n
    cot = rng.standard_normal((n, 3))
    lv = psr.Leaves.build(pos, mass, L, r_s, r_c, max_leaf=max_leaf).upload()
    o = psr.Options(precision=psr.PSR_FP64)
    acc = lv.forces(o)
    gx, gm = (g.cpu().numpy() for g in lv.adjoint(torch.tensor(cot), o))
    part = torch.zeros_like(acc)
    for k in range(2):
        lv.forces(psr.Options(precision=psr.PSR_FP64, shard_count=2, shard_index=k), out=part)
    assert torch.equal(acc, part)
    lv.check()
    ref = oracle.forces(pos, mass, L, r_s, r_c, 1.0)
    ref = ref[0] if isinstance(ref, tuple) else ref
    ox, om = oracle.adjoint(pos, mass, cot, L, r_s, r_c, 1.0)[:2]
    assert _rms(acc.cpu().numpy(), ref) < 1e-13
    assert _rms(gx, ox) < 1e-13 and _rms(gm, om) < 1e-13


@pytest.mark.parametrize("f", [1e-6, 0.01, 0.5, 1 - 1e-15, 1.0, 1 + 1e-15])
def test_fp64_pair_and_strict_cutoff(f):
    L, r_c, r_s = 64.0, 8.0, 2.0
    pos = np.array([[16.0, 16.0, 16.0], [16.0 + f * r_c, 16.0, 16.0]])
    lv = psr.Leaves.build(pos, np.array([0.5, 0.25]), L, r_s, r_c).upload()
    acc = lv.forces(psr.Options(precision=psr.PSR_FP64)).cpu().numpy()
    r = pos[1, 0] - pos[0, 0]
    want = oracle.T(np.array([r / (2 * r_s)]))[0] / r ** 2 if r < r_c else 0.0
    np.testing.assert_allclose(acc[:, 0], [0.25 * want, -0.5 * want], rtol=2e-15)
    assert np.all(acc[:, 1:] == 0.0)


@pytest.mark.parametrize("r_s", [1e-6, 1.1e-7, 0.9e-7, 0.5e-7, 1e-9, 1e-13])
@pytest.mark.parametrize("device", [False, True])
def test_fp64_cutoff_far_beyond_the_table(r_s, device):
    """r_s so far below r_c that a distance in node spacings passes 2^31 and 2^32: those pairs
    have T = 0, and the close ones (a neighbour at 0.4 r_s) keep theirs.  Coordinates are off by
    2^-53 L against 0.4 r_s, so the tolerance is four of those."""
    rng = np.random.default_rng(2)
    n, L, r_c = 600, 10.0, 4.5
    pos = rng.random((n, 3)) * L
    pos[1::2] = np.mod(pos[::2] + np.array([0.4 * r_s, 0.0, 0.0]), L)
    mass, cot = rng.uniform(0.5, 1.5, n), rng.standard_normal((n, 3))
    o = psr.Options(precision=psr.PSR_FP64)
    if device:
        lv = psr.Leaves.device_build(torch.tensor(pos, device="cuda"), torch.tensor(mass, device="cuda"), L, r_s, r_c)
    else:
        lv = psr.Leaves.build(pos, mass, L, r_s, r_c).upload()
    acc = lv.forces(o).cpu().numpy()
    gx, gm = (g.cpu().numpy() for g in lv.adjoint(torch.tensor(cot), o))
    lv.check()
    ref = oracle.forces(pos, mass, L, r_s, r_c, 1.0)
    ref = ref[0] if isinstance(ref, tuple) else ref
    ox, om = oracle.adjoint(pos, mass, cot, L, r_s, r_c, 1.0)[:2]
    tol = 1e-13 + 4 * 2.0 ** -53 * L / (0.4 * r_s)
    assert _rms(acc, ref) < tol and _rms(gx, ox) < 3 * tol and _rms(gm, om) < tol


@pytest.mark.parametrize("x_c", [2.25, 5.3, 5.4, 9.0, 12.0, 14.0])
def test_fp64_pairs_over_all_separations(x_c):
    """Isolated pairs from x = 1e-3 x_c to x_c in units 2 r_s = 1, where x is the separation itself,
    against T and exp(-x^2) in 40 digits: each pair's force and gradients to the roundings of x (r^2's
    and the root's: under 3 x 2^-53, times |x T'/T| < 2 x^2 + 2), 16 roundings of the factors, and
    3e-15 for the folded tables at their far end."""
    mp = pytest.importorskip("mpmath")
    mp.mp.dps = 40
    m, r_c = 10, x_c
    L, x = 3.2 * m * r_c, np.geomspace(1e-3 * x_c, 0.999 * x_c, m ** 3)
    grid = (np.stack(np.meshgrid(*[np.arange(m)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.25) * 3.2 * r_c
    pos = np.empty((2 * m ** 3, 3))
    pos[::2] = pos[1::2] = grid
    pos[1::2, 0] += x
    r = pos[1::2, 0] - pos[::2, 0]
    mass = np.where(np.arange(2 * m ** 3) % 2, 0.25, 0.5)
    cot = np.zeros_like(pos)
    cot[:, 0] = np.where(np.arange(2 * m ** 3) % 2, 2.0, -1.0)
    lv = psr.Leaves.build(pos, mass, L, 0.5, r_c).upload()
    o = psr.Options(precision=psr.PSR_FP64)
    acc = lv.forces(o).cpu().numpy()
    gx, gm = (g.cpu().numpy() for g in lv.adjoint(torch.tensor(cot), o))
    Q = [mp.e ** (-mp.mpf(float(v)) ** 2) for v in r]
    T = [mp.erfc(mp.mpf(float(v))) + 2 / mp.sqrt(mp.pi) * mp.mpf(float(v)) * q for v, q in zip(r, Q)]
    f = np.array([float(t / mp.mpf(float(v)) ** 2) for t, v in zip(T, r)])
    # longitudinal g + r g'(r) = -2 g - Q / (2 sqrt(pi) r_s^3)
    k = np.array([float(-2 * t / mp.mpf(float(v)) ** 3 - 4 / mp.sqrt(mp.pi) * q) for t, q, v in zip(T, Q, r)])
    tol = (16 + 3 * (2 * r * r + 2)) * 2.0 ** -53 + np.where(r > 3.0, 3e-15, 0.0)
    for got, want in ((acc[::2, 0], 0.25 * f), (acc[1::2, 0], -0.5 * f),
                      (gm[::2], -2.0 * f), (gm[1::2], -1.0 * f),
                      (gx[::2, 0], k * (0.5 * 2.0 + 0.25 * 1.0)), (gx[1::2, 0], -k * (0.5 * 2.0 + 0.25 * 1.0))):
        assert np.all(np.abs(got / want - 1.0) < tol), float(np.max(np.abs(got / want - 1.0) / tol))
