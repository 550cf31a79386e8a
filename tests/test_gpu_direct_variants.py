"""GPU: the direct-read steps of matrices held in L2, by row length and size,
bit for bit against the staged steps."""
import numpy as np
import pytest

import synth
from gpu_util import dev_csr, ppg_or_skip, random_csr, to_dev

pytestmark = pytest.mark.gpu

ROOTS = np.array([6.0, 5 + 2j, 5 - 2j, 4.5, 7 + 0.5j, 7 - 0.5j, 6.5], dtype=complex)
MATRICES = {
    "two_ctas_per_sm": lambda: synth.cd2d(182, 0.7),            # five entries a row
    "nine_ctas_per_sm": lambda: synth.cd2d(401, 0.7),
    "ten_and_eleven": lambda: synth.cd2d(443, 0.7),             # where even placement ends
    "seven_entries": lambda: synth.cd3d(36, (0.8, 0.4, 0.2)),
    "seven_entries_one_wave": lambda: synth.cd3d(53, (0.8, 0.4, 0.2)),
    "seven_entries_more": lambda: synth.cd3d(55, (0.8, 0.4, 0.2)),
    "up_to_thirteen": lambda: random_csr(40007, 8, max_row=13, empty_rows={0, 127, 40006}),
}


@pytest.fixture(scope="module")
def env():
    return ppg_or_skip()


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("name", sorted(MATRICES))
def test_direct_steps_equal_staged_steps(env, name, dtype):
    """A chain of ppg_apply_poly on a matrix held in L2 runs the direct-read
    steps; one product of ppg_spmv at a time on the same matrix runs them
    too, and a block-diagonal matrix too large for L2 runs the staged ones."""
    p, torch = env
    tdt = torch.float64 if dtype == "f64" else torch.float32
    H = MATRICES[name]()
    A = dev_csr(p, torch, H, dtype=tdt)
    v = to_dev(torch, np.random.default_rng(1).standard_normal(H.n), tdt)
    R = p.Roots.from_complex(ROOTS)
    # the same rows at the head of a matrix of 1e7 entries and more
    extra = 10_000_000
    big = p.CSR(torch.cat([A.rowptr, A.nnz + torch.arange(1, extra + 1, dtype=torch.int32, device="cuda")]),
                torch.cat([A.colind, A.n + torch.arange(extra, dtype=torch.int32, device="cuda")]),
                torch.cat([A.vals, torch.full((extra,), 5.0, dtype=tdt, device="cuda")]))
    vb = torch.cat([v, torch.ones(extra, dtype=tdt, device="cuda")])
    assert torch.equal(p.apply_poly(A, R, v), p.apply_poly(big, R, vb)[: A.n])
    assert torch.equal(p.apply_phi(A, R, v), p.apply_phi(big, R, vb)[: A.n])
    assert torch.equal(p.spmv(A, v), p.spmv(big, vb)[: A.n])
