"""P2M and L2P share a cell between a few lanes: cells of fewer particles than
lanes (none, one, two, three), of remainders, and cell counts that leave the last
block partly empty, element by element against the FP64 oracle operators.

Bounds: P2M is a sum of at most 70 positive-mass FP32 terms, each of relative
error below 8 roundings (2^-24 each); 78 x 2^-24 = 4.7e-6 of the sum of
magnitudes.  L2P is an FP32 sum of at most 83 coefficient terms with products
of up to 6 factors: 100 x 2^-24 = 6e-6 of the sum of magnitudes; the
coefficients reach the kernel in FP32 as they are given to the oracle.
"""
import numpy as np
import pytest

from oracle import fmm as ofmm

psr = pytest.importorskip("paper_2107_14008_gb300")
from paper_2107_14008_gb300 import capi  # noqa: E402


def _ragged(ncell, seed):
    rng = np.random.default_rng(seed)
    cnt = np.concatenate([np.arange(10), [31, 32, 33, 70], rng.integers(0, 40, ncell)])[:ncell]
    first = np.concatenate([[0], np.cumsum(cnt)]).astype(np.int64)
    centres = rng.uniform(0, 10, (ncell, 3))
    pos = np.repeat(centres, cnt, axis=0) + rng.uniform(-0.4, 0.4, (first[-1], 3))
    return rng, centres, pos, rng.uniform(0.5, 1.5, first[-1]), first


@pytest.mark.gpu
@pytest.mark.parametrize("p,ncell", [(1, 2), (2, 14), (4, 33), (6, 67)])
def test_cells_of_any_count_match_the_oracle(p, ncell):
    import torch
    h, G, L = 0.8, 1.3, 1000.0
    rng, centres, pos, mass, first = _ragged(ncell, 10 * p + ncell)
    nc, idx = capi.psr_fmm_ncoef(p), ofmm.multi_indices(p)
    stream = torch.cuda.current_stream().cuda_stream
    f, x, m, z = (torch.tensor(a, device="cuda") for a in (first, pos, mass, centres))
    M = torch.full((ncell, nc), 7.0, dtype=torch.float32, device="cuda")
    capi.psr_fmm_p2m(p, h, len(pos), ncell, f.data_ptr(), x.data_ptr(), m.data_ptr(),
                     z.data_ptr(), M.data_ptr(), stream)
    M = M.double().cpu().numpy()
    Lg = rng.standard_normal((ncell, nc)).astype(np.float32)
    lg = torch.tensor(Lg, device="cuda")
    acc = torch.full((len(pos), 3), 7.0, dtype=torch.float32, device="cuda")
    capi.psr_fmm_l2p(p, h, capi.psr_box(L, 1.2, 5.4, G), ncell, f.data_ptr(), x.data_ptr(),
                     z.data_ptr(), lg.data_ptr(), acc.data_ptr(), 0, stream)
    acc = acc.double().cpu().numpy()
    scale_m = np.array([h ** -sum(n) for n in idx])
    scale_l = np.array([h ** -(sum(n) + 1) for n in idx])
    for c in range(ncell):
        sl = slice(first[c], first[c + 1])
        if sl.start == sl.stop:
            assert np.all(M[c] == 0.0), c
            continue
        d = np.abs(pos[sl] - centres[c])
        ref = ofmm.p2m(pos[sl], mass[sl], centres[c], p) * scale_m
        mag = ofmm.p2m(centres[c] - d, mass[sl], centres[c], p) * scale_m
        assert np.all(np.abs(M[c] - ref) <= 4.7e-6 * mag), c
        ref = ofmm.l2p(Lg[c].astype(np.float64) * scale_l, centres[c], pos[sl], p, G)
        mag = ofmm.l2p(np.abs(Lg[c].astype(np.float64)) * scale_l, centres[c], centres[c] + d, p, G)
        assert np.all(np.abs(acc[sl] - ref) <= 6e-6 * np.abs(mag)), c
