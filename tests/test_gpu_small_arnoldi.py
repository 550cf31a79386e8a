"""GPU: a small system's Arnoldi step in one launch: the residual after one
cycle and the Hessenberg matrix against NumPy's."""
import numpy as np
import pytest

import synth
from gpu_util import dev_csr, ppg_or_skip, random_csr, to_dev

pytestmark = pytest.mark.gpu

# name -> (matrix, cycle lengths); rows are dealt to 16 blocks in multiples of 32
SYSTEMS = {
    "thirty_three_rows": (lambda: synth.diag_csr(1.0 + np.arange(33.0)), (1, 4, 5, 9)),
    "last_block_short": (lambda: synth.diag_csr(1.0 + np.arange(481.0)), (8, 33)),
    "blocks_without_rows": (lambda: random_csr(40, 3, diag=30.0), (1, 2, 3)),
    "half_blocks": (lambda: synth.cd2d(64, 0.5), (16, 63, 64, 65, 70)),     # 256 rows a block
    "whole_blocks": (lambda: synth.cd2d(65, 0.5), (17, 66)),                # 288 rows a block
    "basis_beyond_smem": (lambda: synth.diag_csr(1.0 + np.arange(9000.0)), (30, 32, 34)),
    "end_of_rows": (lambda: synth.diag_csr(1.0 + np.arange(16384.0)), (17, 18, 19)),
    "beyond_rows": (lambda: synth.diag_csr(1.0 + np.arange(16385.0)), (3,)),
}


@pytest.fixture(scope="module")
def env():
    return ppg_or_skip()


def arnoldi(H, v, m):
    M = H.to_scipy()
    V = np.zeros((m + 1, H.n))
    h = np.zeros((m + 1, m))
    V[0] = v / np.linalg.norm(v)
    for j in range(m):
        w = M @ V[j]
        for _ in range(2):
            c = V[: j + 1] @ w
            w = w - c @ V[: j + 1]
            h[: j + 1, j] += c
        h[j + 1, j] = np.linalg.norm(w)
        V[j + 1] = w / h[j + 1, j]
    return V, h


@pytest.mark.parametrize("name", sorted(SYSTEMS))
def test_cycle_residual(env, name):
    """Both residuals are the smallest over the Krylov space up to rounding: of
    the order of eps * ||A|| ||x|| per operation in the m (m + 1) / 2 dot
    products, here below 1e-9 of ||b|| (the largest ||A|| ||x|| / ||b|| is the
    condition number 16,384, times eps times 200).  The estimate from the
    rotations is that residual too."""
    p, torch = env
    make, lengths = SYSTEMS[name]
    H = make()
    A = dev_csr(p, torch, H)
    b = np.random.default_rng(7).standard_normal(H.n)
    for m in lengths:
        x, s = p.solve(A, to_dev(torch, b), m=m, tol=1e-30, max_cycles=1)
        got = np.linalg.norm(b - H.to_scipy() @ x.cpu().numpy()) / np.linalg.norm(b)
        V, h = arnoldi(H, b, m)
        e = np.zeros(m + 1)
        e[0] = 1.0
        y = np.linalg.lstsq(h, e, rcond=None)[0]
        want = np.linalg.norm(e - h @ y)
        assert abs(got - want) < 1e-9
        assert abs(s["est_relres"] - want) < 1e-9


@pytest.mark.parametrize("n", [33, 4096, 4097])
def test_hessenberg(env, n):
    """A random matrix of norm below 12, eight columns: Arnoldi's growth of
    rounding over so few well-separated columns stays below 1e4 eps."""
    p, torch = env
    H = random_csr(n, 5)
    v = np.random.default_rng(8).standard_normal(n)
    _, got = p.build_poly(dev_csr(p, torch, H), 8, to_dev(torch, v), return_hbar=True)
    _, want = arnoldi(H, v, 8)
    np.testing.assert_allclose(got, want, rtol=0, atol=12 * 1e4 * 2.3e-16)
