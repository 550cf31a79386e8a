"""GPU: chains captured into a graph when no L2 set-aside is in place that would do
for them (its size is a limit that cannot change in a capture).  In a process of its
own, whose one earlier call has loaded the library's device code."""
import os
import subprocess
import sys

import pytest

from gpu_util import ppg_or_skip

pytestmark = pytest.mark.gpu

CODE = """
import sys
import numpy as np, torch, synth, paper_1911_07065_gb300 as p
before, kind, side, dtype = int(sys.argv[1]), sys.argv[2], int(sys.argv[3]), getattr(torch, sys.argv[4])
R = p.Roots.from_complex(np.array([5 + 2j, 5 - 2j] * 15))
def system(kind, n):
    H = synth.cd2d(n, 0.5) if kind == "2d" else synth.cd3d(n, (0.8, 0.4, 0.2))
    A = p.CSR.from_host(H.rowptr, H.colind, H.vals, device="cuda", dtype=dtype)
    return A, torch.ones(A.n, dtype=dtype, device="cuda")
A, v = system("2d", before)
p.apply_poly(A, R, v)
A, v = system(kind, side)
y, z, w = (torch.zeros_like(v) for _ in range(3))
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g, stream=torch.cuda.Stream()):
    p.apply_poly(A, R, v, out=y)
    p.apply_phi(A, R, v, out=z)
    p.spmv(A, v, out=w)
for _ in range(2):
    g.replay()
torch.cuda.synchronize()
assert torch.equal(y, p.apply_poly(A, R, v))
assert torch.equal(z, p.apply_phi(A, R, v))
assert torch.equal(w, p.spmv(A, v))
"""


@pytest.fixture(scope="module", autouse=True)
def env():
    return ppg_or_skip()


@pytest.mark.parametrize("dtype", ["float64", "float32"])
@pytest.mark.parametrize("before,kind,side", [
    (20, "2d", 50),      # one cluster
    (50, "2d", 150),     # in L2
    (50, "2d", 700),     # in L2, far above a smaller system's share
    (50, "3d", 150),     # streamed (in FP32 by its diagonals)
    (300, "3d", 150),
])
def test_first_chain_inside_a_capture(before, kind, side, dtype):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.run([sys.executable, "-c", CODE, str(before), kind, str(side), dtype], check=True, cwd=root,
                   timeout=300)
