"""Heavy rows are summed in parts that the row and its box alone decide: a box gives the same forces
and gradients, bit for bit, in a batch and alone, built on the host and on the GPU, whole and in
shards, and whatever the launch's warps and blocks, which decide who forms the parts only.  The sets
are large enough that the boxes' rows have 1, 2, 4 and 8 parts and that the batch shares the rows
of some launches and not of others."""
import numpy as np
import pytest
import torch

import paper_2107_14008_gb300 as psr

pytestmark = pytest.mark.gpu


def _boxes(which, equal):
    rng = np.random.default_rng(4)
    out = []
    sizes = {"small": [(700, 0), (3000, 0), (2500, 900)],
             "mixed": [(600, 0), (9000, 0), (40000, 0), (30000, 4000), (90000, 6000), (120000, 0)]}[which]
    for n, clump in sizes:
        L = 4.0 * n ** (1 / 3)
        pos = rng.random((n, 3)) * L
        pos[:clump] = np.mod(0.3 * L + 0.02 * L * rng.standard_normal((clump, 3)), L)
        mass = np.full(n, 1.0 / n) if equal else rng.uniform(0.5, 1.5, n) / n
        r_s = 1.2 * L / max(8, 2 * round(0.5 * n ** (1 / 3)))
        out.append((pos, mass, L, r_s, 4.5 * r_s, 1.0))
    return out


# the last: tables so large that the totals of rows leave room for fewer warps
OPTS = {"linear": dict(), "kahan": dict(accum=psr.PSR_ACC_KAHAN32), "cubic": dict(interp=psr.PSR_CUBIC),
        "exact": dict(precision=psr.PSR_FP32_EXACT), "fp64": dict(precision=psr.PSR_FP64),
        "large table": dict(interp=psr.PSR_CUBIC, table_n=4096, source_tile=256)}
SHAPES = [dict(), dict(warps_per_block=1), dict(warps_per_block=4, blocks_per_sm=3), dict(warps_per_block=6),
          dict(blocks_per_sm=1), dict(warps_per_block=2, blocks_per_sm=1)]


def _run(lv, cot, kw):
    o = psr.Options(**kw)
    cot = cot if o.fp64 else cot.float()
    acc = lv.forces(o).clone()
    gx, gm = (t.clone() for t in lv.adjoint(cot, o))
    return acc, gx, gm


@pytest.mark.parametrize("which", ["small", "mixed"])
@pytest.mark.parametrize("equal", [True, False])
@pytest.mark.parametrize("max_leaf", [16, 32, 64])
def test_batch_equals_boxes_alone(which, equal, max_leaf):
    boxes = _boxes(which, equal)
    lv = psr.Leaves.build_batch(boxes, max_leaf=max_leaf).upload()
    cots = [torch.tensor(np.random.default_rng(k).standard_normal(b[0].shape), device="cuda")
            for k, b in enumerate(boxes)]
    whole = {k: _run(lv, torch.cat(cots), kw) for k, kw in OPTS.items()}
    lv.check()
    off = 0
    for k, b in enumerate(boxes):
        n = len(b[0])
        one = psr.Leaves.build(*b, max_leaf=max_leaf).upload() if k % 2 else psr.Leaves.device_build(
            torch.tensor(b[0], device="cuda"), torch.tensor(b[1], device="cuda"), *b[2:], max_leaf=max_leaf)
        for name, kw in OPTS.items():
            for u, v in zip(whole[name], _run(one, cots[k], kw)):
                assert torch.equal(u[off:off + n], v), (k, name)
        one.check()
        off += n


@pytest.mark.parametrize("which", ["small", "mixed"])
@pytest.mark.parametrize("name", list(OPTS))
def test_launch_shapes_and_shards_do_not_move_a_bit(which, name):
    boxes = _boxes(which, False)
    cot = torch.tensor(np.random.default_rng(1).standard_normal((sum(len(b[0]) for b in boxes), 3)), device="cuda")
    sets = [(psr.Leaves.build_batch(boxes).upload(), cot)]
    if which == "mixed":  # and one box whose heavy rows have parts
        sets.append((psr.Leaves.build(*boxes[3]).upload(), cot[:len(boxes[3][0])]))
    for lv, c in sets:
        want = _run(lv, c, OPTS[name])
        for kw in SHAPES:
            got = _run(lv, c, dict(OPTS[name], **kw))
            assert all(torch.equal(u, v) for u, v in zip(got, want)), kw
        got = tuple(torch.full_like(t, float("nan")) for t in want)
        for k in range(8):
            o = psr.Options(shard_count=8, shard_index=k, **OPTS[name])
            lv.forces(o, out=got[0])
            lv.adjoint(c if o.fp64 else c.float(), o, got[1], got[2])
        assert all(torch.equal(u, v) for u, v in zip(got, want))
        lv.check()
