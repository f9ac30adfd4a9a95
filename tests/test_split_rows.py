"""Heavy rows shared by the warps of a block (the default kernels on small or strongly clustered
sets): the sums over the parts of a row, combined over the warps, against the oracle and against
the kernels that keep a row on one warp.

Tolerance: the FP32 bound of every path against the oracle, 2e-5 relative RMS; between the two
orders of sums of the same FP32 terms, 2e-6 (chunk partials of at most 256 terms, 2^-24 each)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2107_14008_gb300 as psr

pytestmark = pytest.mark.gpu


def _set(kind):
    rng = np.random.default_rng(11)
    L = 40.0
    if kind == "one_leaf":
        pos = rng.random((23, 3)) * L
    elif kind == "few":  # fewer leaves than warps: every row is shared
        pos = rng.random((3000, 3)) * L
    else:  # enough leaves that only the dense clump's rows are shared
        pos = np.concatenate([rng.random((110000, 3)) * L, 8.0 + 0.25 * rng.standard_normal((4000, 3))])
    n = len(pos)
    return pos, np.full(n, 1.0 / n), L, 0.5, 2.25


def _rms(a, b):
    return float(np.sqrt(((a - b) ** 2).sum() / (b ** 2).sum()))


@pytest.mark.parametrize("kind", ["one_leaf", "few", "clump"])
@pytest.mark.parametrize("max_leaf", [8, 32, 64])
@pytest.mark.parametrize("kw", [dict(), dict(accum=psr.PSR_ACC_KAHAN32), dict(interp=psr.PSR_CUBIC),
                                dict(precision=psr.PSR_FP32_EXACT), dict(warps_per_block=1),
                                dict(warps_per_block=6, source_tile=64)])
def test_shared_rows_match_oracle_and_single_warp_rows(kind, max_leaf, kw):
    pos, mass, L, r_s, r_c = _set(kind)
    if kind == "one_leaf":
        r_s, r_c = 4.0, 18.0
    lv = psr.Leaves.build(pos, mass, L, r_s, r_c, max_leaf=max_leaf).upload()
    acc = lv.forces(psr.Options(**kw))
    assert torch.equal(acc, lv.forces(psr.Options(**kw)))
    one = lv.forces(psr.Options(kernel=psr.PSR_KERNEL_SCALAR, **kw)).double().cpu().numpy()
    part = torch.zeros_like(acc)
    for k in range(3):
        lv.forces(psr.Options(shard_count=3, shard_index=k, **kw), out=part)
    assert torch.equal(acc, part)
    acc = acc.double().cpu().numpy()
    cot = np.random.default_rng(3).standard_normal(pos.shape)
    gx, gm = (g.double().cpu().numpy() for g in lv.adjoint(torch.tensor(cot), psr.Options(**kw)))
    hx, hm = (g.double().cpu().numpy() for g in
              lv.adjoint(torch.tensor(cot), psr.Options(kernel=psr.PSR_KERNEL_SCALAR, **kw)))
    lv.check()
    assert _rms(acc, one) < 2e-6 and _rms(gx, hx) < 2e-6 and _rms(gm, hm) < 2e-6
    if kind != "clump":
        ref = oracle.forces(pos, mass, L, r_s, r_c, 1.0)
        ref = ref[0] if isinstance(ref, tuple) else ref
        ox, om = oracle.adjoint(pos, mass, cot, L, r_s, r_c, 1.0)[:2]
        assert _rms(acc, ref) < 2e-5 and _rms(gx, ox) < 2e-5 and _rms(gm, om) < 2e-5


def test_device_built_schedule_marks_the_same_rows():
    pos, mass, L, r_s, r_c = _set("clump")
    a = psr.Leaves.build(pos, mass, L, r_s, r_c).upload()
    b = psr.Leaves.device_build(torch.tensor(pos, device="cuda"), torch.tensor(mass, device="cuda"),
                                L, r_s, r_c)
    assert torch.equal(a.forces(), b.forces())


@pytest.mark.parametrize("x_c", [0.4, 2.25, 2.5, 2.6, 4.5, 4.6])
@pytest.mark.parametrize("accum", [psr.PSR_ACC_FP64, psr.PSR_ACC_KAHAN32])
def test_exact_precision_by_the_fine_table_and_by_erfc(x_c, accum):
    """PSR_FP32_EXACT under the default kernel (a fine cubic table up to x_c = 4.5) against the
    kernel that calls erfcf and expf, and the oracle.  T of both is within a few FP32 roundings:
    1e-6 between them, twice the roundings of a weight (4 x 2^-24 each), summed incoherently."""
    pos, mass, L, _, r_c = _set("few")
    r_c = 6.0
    r_s = r_c / (2.0 * x_c)
    cot = np.random.default_rng(3).standard_normal(pos.shape)
    lv = psr.Leaves.build(pos, mass, L, r_s, r_c).upload()
    a, b = (lv.forces(psr.Options(precision=psr.PSR_FP32_EXACT, accum=accum, kernel=k)).double().cpu().numpy()
            for k in (psr.PSR_KERNEL_AUTO, psr.PSR_KERNEL_SCALAR))
    ga, gb = (lv.adjoint(torch.tensor(cot), psr.Options(precision=psr.PSR_FP32_EXACT, accum=accum, kernel=k))
              for k in (psr.PSR_KERNEL_AUTO, psr.PSR_KERNEL_SCALAR))
    ref = oracle.forces(pos, mass, L, r_s, r_c, 1.0)
    ref = ref[0] if isinstance(ref, tuple) else ref
    assert _rms(a, b) < 1e-6 and _rms(a, ref) < 2e-5
    for u, v in zip(ga, gb):
        assert _rms(u.double().cpu().numpy(), v.double().cpu().numpy()) < 1e-6
