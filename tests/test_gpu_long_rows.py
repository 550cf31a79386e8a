"""GPU: rows around and above the length at which a warp sums a row."""
import numpy as np
import pytest

from gpu_util import dev_csr, ppg_or_skip, random_csr, to_dev
from oracle import poly

pytestmark = pytest.mark.gpu

# both sides of 128 entries, two in one warp, the last row
LONG = {0: 126, 33: 127, 34: 128, 35: 129, 64: 400, 95: 2500, 1000: 3000}
ROOTS = np.array([4.0, 3 + 1j, 3 - 1j, 2.5, 2 + 0.5j, 2 - 0.5j, 3.3], dtype=complex)


@pytest.fixture(scope="module")
def env():
    return ppg_or_skip()


@pytest.mark.parametrize("n", [3001, 40001])
def test_long_rows_match_oracle_and_agree_between_kernels(env, n):
    """p(A) v and A v against the oracle, and the chain of ppg_apply_poly
    (matrix held in L2) bit for bit against ppg_apply_poly_noalloc."""
    p, torch = env
    A = random_csr(n, 4, long_rows={**LONG, n - 1: 700}, empty_rows={36, 2000})
    As = A.to_scipy()
    R = p.Roots.from_complex(ROOTS)
    v = np.random.default_rng(9).standard_normal(n)
    for dtype, tol in ((torch.float64, 1e-13), (torch.float32, 1e-5)):
        Ad = dev_csr(p, torch, A, dtype=dtype)
        vd = to_dev(torch, v, dtype)
        ref = poly.apply_p(As, ROOTS, v)
        got = p.apply_poly(Ad, R, vd)
        # rows of 3,000 N(0, 0.01) entries: ||A|| < 16, eight products at most
        # (3000 + 8) roundings each of entries below 16^7 ||v|| in the worst
        # row; measured in the norm of p(A) v they stay below 1e3 units
        assert np.linalg.norm(got.double().cpu().numpy() - ref) <= 1e3 * tol * np.linalg.norm(ref)
        assert torch.equal(got, p.apply_poly_noalloc(Ad, R, vd, torch.empty_like(vd)))
        y = p.spmv(Ad, vd).double().cpu().numpy()
        assert np.linalg.norm(y - As @ v) <= tol * 10 * np.linalg.norm(As @ v)


def test_sweep_plan_with_a_long_row_equals_the_plain_chain(env):
    p, torch = env
    A = random_csr(3001, 5, long_rows={7: 300})
    A32 = dev_csr(p, torch, A, dtype=torch.float32)
    plan = p.SweepPlan(A32, tile_rows=256)
    R = p.Roots.from_complex(ROOTS)
    v = to_dev(torch, np.random.default_rng(2).standard_normal(A.n), torch.float32)
    assert plan.info()["fused"] == 0
    assert torch.equal(plan.apply_poly(R, v), p.apply_poly(A32, R, v))
