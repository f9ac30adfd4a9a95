"""The GPU builder's single-pass sort, scans and sliding-maximum leaf levels at the sizes where
their tiles end: one block's sort (8192 items), whole and partial tiles of 4096, one and several
scan tiles, windows of every leaf size.  The workspace has to be the host builder's bit for bit."""
import numpy as np
import pytest
import torch

import paper_2107_14008_gb300 as psr

pytestmark = pytest.mark.gpu


def _same(pos, mass, L, r_s, r_c, **kw):
    h = psr.Leaves.build(pos, mass, L, r_s, r_c, **kw)
    d = psr.Leaves.device_build(torch.tensor(pos, device="cuda"),
                                None if mass is None else torch.tensor(mass, device="cuda"), L, r_s, r_c, **kw)
    d.check()
    a, b = h.host_arrays(), d.device_arrays()
    for k in ("pf", "leaf", "lcen", "rowptr", "pairs", "items", "pd"):
        assert np.array_equal(np.asarray(a[k]).view(np.uint8), np.asarray(b[k]).view(np.uint8)), k
    assert np.array_equal(h.perm, d.perm)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 255, 256, 257, 4095, 4096, 4097, 8191, 8192, 8193, 12288, 12289,
                               40961])
def test_sizes_at_tile_ends(n):
    rng = np.random.default_rng(n)
    L = 10.0
    _same(rng.random((n, 3)) * L, rng.random(n), L, 0.2, 0.9)


@pytest.mark.parametrize("max_leaf", [1, 2, 3, 7, 16, 31, 33, 63, 64])
@pytest.mark.parametrize("pack", [True, False])
def test_leaf_sizes_with_coincident_and_clustered_particles(max_leaf, pack):
    rng = np.random.default_rng(max_leaf)
    L = 10.0
    pos = np.concatenate([rng.random((3000, 3)) * L, np.full((150, 3), 3.7), np.full((max_leaf, 3), 6.1),
                          np.full((max_leaf + 1, 3), 8.2), 5.0 + 1e-4 * rng.standard_normal((2000, 3))])
    _same(pos, None, L, 0.2, 0.9, max_leaf=max_leaf, pack=pack)


@pytest.mark.parametrize("scale", [1.0, 1e-6, 1e6])
def test_small_cutoffs_leave_the_decision_to_fp64(scale):
    """r_c far below the FP32 spacing of the coordinates' range times 2^4: the walk's FP32 bounds
    decide little and the host's FP64 test the rest."""
    rng = np.random.default_rng(3)
    L = 1000.0 * scale
    pos = rng.random((4000, 3)) * L
    pos[1::2] = pos[::2] + rng.uniform(-1, 1, (2000, 3)) * 1e-3 * scale
    _same(pos, None, L, 1e-4 * scale, 4.5e-4 * scale, max_leaf=1)
