"""GPU: a small system's chain in one launch against the step-by-step chain,
bit for bit."""
import os
import subprocess
import sys

import numpy as np
import pytest

import synth
from gpu_util import dev_csr, ppg_or_skip, random_csr, to_dev

pytestmark = pytest.mark.gpu

MATRICES = {
    "one_row": lambda: synth.diag_csr(np.array([3.0])),
    "thirty_three_rows": lambda: random_csr(33, 1),
    "grid_50": lambda: synth.cd2d(50, 0.5),
    "grid_103": lambda: synth.cd2d(103, 0.5),          # 10,609 rows: the end of the FP64 range
    "grid_128": lambda: synth.cd2d(128, 0.5),          # 16,384 rows: the end of the FP32 range
    "two_rows_a_thread": lambda: synth.diag_csr(3.0 + np.arange(8193) / 8193),
    "cube_19": lambda: synth.cd3d(19, (0.8, 0.4, 0.2)),
    "long_and_empty": lambda: random_csr(3001, 2, long_rows={0: 128, 5: 129, 6: 2000, 700: 900, 3000: 300},
                                         empty_rows={1, 17, 2999}),
}
ROOTS = {
    "real": np.array([6.0, 5.0, 7.5, 4.0]),
    "pairs": np.array([5 + 2j, 5 - 2j, 7 + 1j, 7 - 1j]),
    "pair_then_real": np.array([6.0, 5 + 2j, 5 - 2j, 3.3]),
    "degree_two": np.array([5 + 1j, 5 - 1j]),
    "long": np.array([5.5 + 0.01 * k for k in range(60)]),
}


@pytest.fixture(scope="module")
def env():
    return ppg_or_skip()


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("name", sorted(MATRICES))
def test_one_launch_equals_steps(env, name, dtype):
    """The same rows as the head of a block-diagonal matrix of 40,000 rows run
    step by step."""
    p, torch = env
    tdt = torch.float64 if dtype == "f64" else torch.float32
    H = MATRICES[name]()
    A = dev_csr(p, torch, H, dtype=tdt)
    extra = 40000 - H.n
    big = p.CSR(torch.cat([A.rowptr, A.nnz + torch.arange(1, extra + 1, dtype=torch.int32, device="cuda")]),
                torch.cat([A.colind, A.n + torch.arange(extra, dtype=torch.int32, device="cuda")]),
                torch.cat([A.vals, torch.full((extra,), 5.0, dtype=tdt, device="cuda")]))
    v = to_dev(torch, np.random.default_rng(1).standard_normal(H.n), tdt)
    vb = torch.cat([v, torch.ones(extra, dtype=tdt, device="cuda")])
    for roots in ROOTS.values():
        R = p.Roots.from_complex(roots)
        assert torch.equal(p.apply_poly(A, R, v), p.apply_poly(big, R, vb)[: A.n])
        assert torch.equal(p.apply_phi(A, R, v), p.apply_phi(big, R, vb)[: A.n])


def test_one_launch_inside_a_graph_and_on_two_streams(env):
    p, torch = env
    A = dev_csr(p, torch, synth.cd2d(60, 0.5))
    R = p.Roots.from_complex(ROOTS["long"])
    v = to_dev(torch, np.random.default_rng(2).standard_normal(A.n))
    ref = p.apply_poly(A, R, v)
    y = torch.empty_like(v)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        p.apply_poly(A, R, v, out=y)
    g.replay()
    outs = []
    for _ in range(4):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            outs.append(p.apply_poly(A, R, v))
    torch.cuda.synchronize()
    assert torch.equal(y, ref) and all(torch.equal(o, ref) for o in outs)


def test_capture_of_a_larger_system_after_a_small_one(env):
    """In a fresh process: the small system's call leaves the L2 share that the
    larger one's chain needs, which could not be set inside a capture."""
    code = """
import numpy as np, torch, synth, paper_1911_07065_gb300 as p
R = p.Roots.from_complex(np.array([5 + 2j, 5 - 2j] * 15))
def system(n):
    H = synth.cd2d(n, 0.5)
    A = p.CSR.from_host(H.rowptr, H.colind, H.vals, device="cuda")
    return A, torch.ones(A.n, dtype=torch.float64, device="cuda")
A, v = system(50)
p.apply_poly(A, R, v)
A, v = system(150)
y = torch.empty_like(v)
torch.cuda.synchronize()
g = torch.cuda.CUDAGraph()
with torch.cuda.graph(g, stream=torch.cuda.Stream()):
    p.apply_poly(A, R, v, out=y)
g.replay()
assert torch.equal(y, p.apply_poly(A, R, v))
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.run([sys.executable, "-c", code], check=True, cwd=root, timeout=120)
