"""CUDA graphs and the interpolation tables: a replayed graph reads its own table whatever other
precision ran on the handle in between, and a call outside a capture does not take a table that
the capture only recorded.  All comparisons are bit for bit with the same call made eagerly."""
import numpy as np
import pytest
import torch

import paper_2107_14008_gb300 as psr

pytestmark = pytest.mark.gpu

EXACT = psr.Options(precision=psr.PSR_FP32_EXACT)
FP64 = psr.Options(precision=psr.PSR_FP64)
LINEAR = psr.Options()
SCALAR = psr.Options(kernel=psr.PSR_KERNEL_SCALAR)
CUBIC = psr.Options(interp=psr.PSR_CUBIC)
ALL = {"exact": EXACT, "fp64": FP64, "linear": LINEAR, "scalar": SCALAR, "cubic": CUBIC}


def _set():
    rng = np.random.default_rng(8)
    n, L = 20000, 40.0
    pos = np.concatenate([rng.random((18000, 3)) * L, 9.0 + 0.5 * rng.standard_normal((2000, 3))])
    return np.mod(pos, L), rng.uniform(0.5, 1.5, n), torch.tensor(rng.standard_normal((n, 3))), (L, 0.5, 2.25)


class Calls:
    """forces and adjoint of one handle, into kept buffers, by the name of their options."""

    def __init__(self):
        pos, mass, self.cot, box = _set()
        self.lv = psr.Leaves.build(pos, mass, *box)
        # what the workspace's memory then holds
        torch.full((int(self.lv.info.device_bytes),), 0x5A, dtype=torch.uint8, device="cuda")
        self.lv.upload()
        self.cot = self.cot.cuda()
        self.cot32 = self.cot.float()

    def __call__(self, what, name):
        o = ALL[name]
        if what == "forces":
            return (self.lv.forces(o),)
        return tuple(self.lv.adjoint(self.cot if o.fp64 else self.cot32, o))

    def capture(self, what, name):
        o = ALL[name]
        out = [torch.empty_like(t) for t in Calls()(what, name)]
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            if what == "forces":
                self.lv.forces(o, out=out[0])
            else:
                self.lv.adjoint(self.cot if o.fp64 else self.cot32, o, *out)
        for t in out:
            t.zero_()
        return g, out


def _same(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("what", ["forces", "adjoint"])
@pytest.mark.parametrize("kept", ["exact", "fp64", "linear"])
def test_replay_after_other_precisions(what, kept):
    c = Calls()
    want = [t.clone() for t in c(what, kept)]  # warm: the graph records no table
    g, out = c.capture(what, kept)
    for name in ALL:
        if name == "cubic" and (what, kept) == ("adjoint", "linear"):
            continue  # the two tables share their place
        c("forces", name)
        c("adjoint", name)
        g.replay()
        torch.cuda.synchronize()
        assert _same(out, want), name
    c.lv.check()


@pytest.mark.parametrize("what", ["forces", "adjoint"])
@pytest.mark.parametrize("name", list(ALL))
def test_eager_call_between_a_first_capture_and_its_replay(what, name):
    want = [t.clone() for t in Calls()(what, name)]
    c = Calls()
    g, out = c.capture(what, name)
    assert _same(c(what, name), want)  # not yet replayed: the recorded table has not been built
    g.replay()
    torch.cuda.synchronize()
    assert _same(out, want)
    c.lv.check()


def test_eager_calls_after_replays_that_write_another_table():
    want = {n: Calls()("forces", n)[0].clone() for n in ("cubic", "scalar")}
    c = Calls()
    g, out = c.capture("forces", "cubic")  # records the cubic table
    for _ in range(2):
        assert torch.equal(c("forces", "scalar")[0], want["scalar"])
        g.replay()
        assert torch.equal(c("forces", "scalar")[0], want["scalar"])
        g.replay()
        assert torch.equal(c("forces", "cubic")[0], want["cubic"]) and torch.equal(out[0], want["cubic"])
    g2, out2 = c.capture("forces", "scalar")  # a second graph on the same place
    for _ in range(2):
        g.replay()
        g2.replay()
        assert torch.equal(c("forces", "cubic")[0], want["cubic"])
        assert torch.equal(out2[0], want["scalar"]) and torch.equal(out[0], want["cubic"])
    c.lv.check()
