"""The forward's core form of the linear table (1/r^3 minus an interpolated smooth part): taken
from 1024 intervals on and for x_c <= 3.5, with scalar streams and with packed pairs.

Tolerances: FP32 forces against the oracle 2e-5 relative RMS, the bound of every FP32 path.  A
single pair at distance r has a weight T/r^3 whose T is off by at most the table's interpolation
error (below 2e-6 on this range) plus four FP32 roundings of terms up to 1/r^3 (2.4e-7 each with
the 2^-22.9 of rsqrt): 4e-6 in units of G m / r^2, and exactly zero at and beyond the cutoff."""
import numpy as np
import pytest

import oracle
import paper_2107_14008_gb300 as psr

pytestmark = pytest.mark.gpu
KERNELS = [psr.PSR_KERNEL_AUTO, psr.PSR_KERNEL_SCALAR, psr.PSR_KERNEL_PACKED]


def _forces(pos, mass, L, r_s, r_c, max_leaf=32, **kw):
    lv = psr.Leaves.build(pos, mass, L, r_s, r_c, max_leaf=max_leaf).upload()
    acc = lv.forces(psr.Options(**kw)).double().cpu().numpy()
    lv.check()
    return acc


@pytest.mark.parametrize("kernel", KERNELS)
@pytest.mark.parametrize("equal", [True, False])
@pytest.mark.parametrize("table_n,x_c", [(512, 2.25), (1024, 0.3), (1024, 2.25), (1024, 3.5),
                                         (1024, 3.6), (4096, 2.25), (8192, 3.0)])
def test_matches_oracle_over_tables_and_cutoffs(kernel, equal, table_n, x_c):
    rng = np.random.default_rng(7)
    n, L = 1501, 50.0
    pos = rng.random((n, 3)) * L
    pos[:300] = 10.0 + 2.0 * rng.standard_normal((300, 3))
    mass = np.full(n, 1.0 / n) if equal else rng.uniform(0.2, 2.0, n) / n
    r_c = 12.0
    r_s = r_c / (2.0 * x_c)
    ref = oracle.forces(pos, mass, L, r_s, r_c, 1.0)
    ref = ref[0] if isinstance(ref, tuple) else ref
    acc = _forces(pos, mass, L, r_s, r_c, table_n=table_n, kernel=kernel)
    tol = 2e-5 if table_n >= 1024 else 5e-5  # a 512 chord table is off by 3e-6 in T
    assert np.sqrt(((acc - ref) ** 2).sum() / (ref ** 2).sum()) < tol


@pytest.mark.parametrize("kernel", KERNELS)
@pytest.mark.parametrize("f", [1e-3, 0.03, 0.3, 0.7, 0.99, 1 - 1e-5, 1 + 1e-5, 1.01, 1.3])
def test_single_pair_and_hard_cutoff(kernel, f):
    L, r_s = 64.0, 2.0
    r_c = 4.5 * r_s
    r = f * r_c
    d = np.array([0.6, 0.64, 0.48]) * r
    pos = np.array([[20.0, 21.0, 22.0], [20.0, 21.0, 22.0] + d])
    mass = np.array([0.5, 0.5])
    acc = _forces(pos, mass, L, r_s, r_c, kernel=kernel)
    if f > 1:
        assert np.all(acc == 0.0)
        return
    want = 0.5 * oracle.T(np.array([r / (2 * r_s)]))[0] * d / r ** 3
    # plus the leaf-local coordinates' rounding: 2^-24 of the leaf cell, at most r_c here
    slack = 4e-6 + 6.0 * 2.0 ** -24 * r_c / r
    assert np.abs(acc[0] - want).max() <= slack * 0.5 / r ** 2
    assert np.abs(acc[1] + want).max() <= slack * 0.5 / r ** 2


@pytest.mark.parametrize("kernel", KERNELS)
def test_coincident_particles_give_zero(kernel):
    pos = np.full((40, 3), 7.0)
    assert np.all(_forces(pos, np.full(40, 0.1), 64.0, 2.0, 9.0, kernel=kernel) == 0.0)
