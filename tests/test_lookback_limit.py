"""A look-back of the GPU builder's sorts or scans that runs out ends the build with PSR_E_DEVICE:
nothing is read or written out of range and the context stays usable.  The builder is compiled once
more with a limit of no polls, so that every wait runs out, and used in a process of its own."""
import os
import subprocess
import sys

import pytest

from paper_2107_14008_gb300 import build as b

pytestmark = pytest.mark.gpu

PROGRAM = """
import numpy as np, torch
import paper_2107_14008_gb300 as psr
from paper_2107_14008_gb300 import capi

L, r_s, r_c = 10.0, 0.2, 0.9
rng = np.random.default_rng(1)
pos = torch.tensor(rng.random((300000, 3)) * L, device="cuda")
# one tile of a scan (no look-back), then several tiles of the scans, of the sorts, and of all
for n, theta in ((4096, None), (4097, None), (8193, None), (20000, 0.5), (300000, None), (4000, 0.5)):
    try:
        lv = psr.Leaves.device_build(pos[:n].contiguous(), None, L, r_s, r_c, theta=theta)
        lv.forces()
        lv.check()
        code = 0
    except capi.PsrError as e:
        code = e.code
    torch.cuda.synchronize()
    assert code == (0 if n <= 4096 else capi.PSR_E_DEVICE), (n, code)
print("done")
"""


def test_every_look_back_runs_out(tmp_path):
    b.build()
    obj, lib = str(tmp_path / "devbuild.o"), str(tmp_path / "libpsr_no_polls.so")
    src = os.path.join(b.SRC, "devbuild.cu")
    subprocess.run([b._nvcc()] + b.ARCH + b.NVCC_FLAGS + ["-DPSR_SPIN_LIMIT=0", "-c", src, "-o", obj], check=True,
                   capture_output=True)
    objs = [os.path.join(b.OUT, f + ".o") for f in b.CU_SOURCES + b.CXX_SOURCES if f != "devbuild.cu"]
    cudalib = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(b._nvcc()))), "lib64")
    subprocess.run([b._nvcc()] + b.ARCH + ["-shared", "-o", lib, obj] + objs +
                   ["-lpthread", "-L" + cudalib, "-lcufft", "-Xlinker", "-rpath=" + cudalib], check=True,
                   capture_output=True)
    r = subprocess.run([sys.executable, "-c", PROGRAM], env=dict(os.environ, PSR_LIB=lib), cwd=b.ROOT,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("done"), r.stdout + r.stderr
