"""Which kernel the differentiable entry point runs: float32 tensors get the options as they are,
float64 tensors PSR_KERNEL_SCALAR in place of the default kernel, and a named kernel is kept.  Bit for
bit against Leaves.forces and Leaves.adjoint, on a set whose rows have parts under the default kernel."""
import numpy as np
import pytest
import torch

import paper_2107_14008_gb300 as psr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("kw", [dict(), dict(precision=psr.PSR_FP32_EXACT), dict(interp=psr.PSR_CUBIC),
                                dict(kernel=psr.PSR_KERNEL_PACKED), dict(kernel=psr.PSR_KERNEL_SCALAR)])
def test_same_bits_as_the_leaf_set(dtype, kw):
    rng = np.random.default_rng(9)
    n, L, r_s, r_c = 3000, 40.0, 0.5, 2.25
    pos = torch.tensor(rng.random((n, 3)) * L, dtype=dtype, device="cuda", requires_grad=True)
    mass = torch.tensor(rng.uniform(0.5, 1.5, n), dtype=dtype, device="cuda", requires_grad=True)
    cot = torch.tensor(rng.standard_normal((n, 3)), dtype=dtype, device="cuda")
    acc = psr.forces(pos, mass, L, r_s, r_c, opts=psr.Options(**kw))
    gx, gm = torch.autograd.grad(acc, (pos, mass), cot)
    named = dict(kw)
    if dtype == torch.float64:
        named.setdefault("kernel", psr.PSR_KERNEL_SCALAR)
    lv = psr.Leaves.device_build(pos.detach().double(), mass.detach().double(), L, r_s, r_c)
    o = psr.Options(**named)
    want = [lv.forces(o), *lv.adjoint(cot.float(), o)]
    assert acc.dtype == gx.dtype == gm.dtype == dtype
    for got, w in zip((acc.detach(), gx, gm), want):
        assert torch.equal(got, w.to(dtype))
