"""GPU: FP32 chains by diagonals against the CSR steps, bit for bit.

ppg_apply_poly builds the diagonal form of a matrix for long FP32 chains.  The
same rows at the head of a matrix with many offsets take the CSR steps.
"""
import numpy as np
import pytest

import synth
from gpu_util import dev_csr, ppg_or_skip, to_dev

pytestmark = pytest.mark.gpu

N = 2_600_003   # not a multiple of any tile; larger than L2; an odd number of tiles


@pytest.fixture(scope="module")
def env():
    return ppg_or_skip()


def _banded(offsets, one_value=(), drop=0.0, empty=(), seed=0, n=N):
    """n rows with entries at `offsets` (inside the matrix), each left out
    with probability `drop`; diagonals in `one_value` have a single value."""
    rng = np.random.default_rng(seed)
    off = np.array(sorted(offsets), dtype=np.int64)
    cols = np.arange(n)[:, None] + off[None, :]
    valid = (cols >= 0) & (cols < n)
    if drop:
        valid &= (rng.random(cols.shape) >= drop) | (off[None, :] == 0)
    valid[list(empty)] = False
    vals = -rng.random(cols.shape) / off.size
    for i, o in enumerate(off):
        if o in one_value:
            vals[:, i] = -0.75 / off.size
        if o == 0:
            vals[:, i] = 4.0 if 0 in one_value else 4.0 + 0.1 * rng.random(n)
    rowptr = np.zeros(n + 1, dtype=np.int64)
    rowptr[1:] = np.cumsum(valid.sum(1))
    return synth.CSRHost(n, rowptr.astype(np.int32), cols[valid].astype(np.int32), vals[valid])


def _csr_steps(p, torch, A, R, v):
    """p(A) v by the CSR steps: 100 rows more, each with an offset of its own."""
    k = torch.arange(100, dtype=torch.int32, device="cuda")
    big = p.CSR(torch.cat([A.rowptr, A.nnz + 1 + k]), torch.cat([A.colind, A.n - 99 * k]),
                torch.cat([A.vals, torch.ones(100, dtype=torch.float32, device="cuda")]))
    return p.apply_poly(big, R, torch.cat([v, v[:100]]))[: A.n]


def _roots():
    """Real roots and pairs around the spectrum, ending in a real root: 34
    factors, 33 matrix products."""
    rng = np.random.default_rng(3)
    out = []
    for i in range(11):
        a, b = 3.2 + 1.6 * rng.random(), 0.1 + 0.3 * rng.random()
        out += [a + 0j, a + 1j * b, a - 1j * b]
    return np.array(out + [4.0 + 0j])


GRID = (-887, -1, 0, 1, 887)
CASES = {
    "one_value_each": dict(offsets=GRID, one_value=GRID),
    "an_even_number_of_tiles": dict(offsets=GRID, one_value=GRID, n=N + 512),
    "some_own_values": dict(offsets=GRID, one_value=(-887, 0, 887)),
    "dropped_entries": dict(offsets=GRID, drop=0.3, empty=(0, 511, 512, N - 1)),
    "close_offsets": dict(offsets=(-17, -16, -2, 0, 3, 18, 19)),
    "nine": dict(offsets=(-900, -899, -898, -1, 0, 1, 898, 899, 900), drop=0.1),
    # more values than a tile's shared memory holds
    "thirteen_apart": dict(offsets=[1000 * k for k in range(-6, 7)]),
    # no such form: too many offsets
    "forty": dict(offsets=list(range(-20, 20)), drop=0.8),
}


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("name", sorted(CASES))
def test_diagonals_equal_csr_steps(env, name, shift):
    p, torch = env
    A = dev_csr(p, torch, _banded(**CASES[name]), dtype=torch.float32)
    R = p.Roots.from_complex(_roots())
    # shift: v and y off a 16-byte boundary
    buf = to_dev(torch, np.random.default_rng(5).standard_normal(A.n + 4), torch.float32)
    v = buf[shift:shift + A.n]
    y = torch.empty(A.n + 4, dtype=torch.float32, device="cuda")[shift:shift + A.n]
    ref = _csr_steps(p, torch, A, R, v)
    p.apply_poly(A, R, v, out=y)
    torch.cuda.synchronize()
    assert torch.isfinite(ref).all()
    assert torch.equal(y, ref)


def test_unsorted_row_keeps_the_csr_steps(env):
    p, torch = env
    H = _banded(GRID)
    k = H.rowptr[400_000]
    H.colind[[k, k + 1]] = H.colind[[k + 1, k]]
    A = p.CSR.from_host(H.rowptr, H.colind, H.vals, dtype=torch.float32, validate=False)
    R = p.Roots.from_complex(_roots())
    v = to_dev(torch, np.random.default_rng(6).standard_normal(N), torch.float32)
    ref = _csr_steps(p, torch, A, R, v)
    assert torch.equal(p.apply_poly(A, R, v), ref)


def test_phi_by_diagonals_against_fp64(env):
    """phi(A) v in FP32 (33 products) against FP64 on the FP32 data.  Every
    factor I - A / theta has norm below 1 here, so each product's rounding,
    at most (5 + 3) 2^-24 of its result, is not amplified: 33 * 8 * 2^-24 =
    1.6e-5 of ||v|| at worst, tolerated up to 1e-4."""
    p, torch = env
    A = dev_csr(p, torch, _banded(GRID, one_value=(0, 1)), dtype=torch.float32)
    R = p.Roots.from_complex(_roots())
    v = to_dev(torch, np.random.default_rng(7).standard_normal(N), torch.float32)
    y = p.apply_phi(A, R, v)
    ref = p.apply_phi(A.astype(torch.float64), R, v.double())
    assert float((y.double() - ref).norm()) <= 1e-4 * float(v.double().norm())


def test_values_seen_by_the_next_call(env):
    """The form is made anew in every call: changed values count."""
    p, torch = env
    A = dev_csr(p, torch, _banded(GRID, one_value=GRID), dtype=torch.float32)
    R = p.Roots.from_complex(_roots())
    v = to_dev(torch, np.random.default_rng(8).standard_normal(N), torch.float32)
    p.apply_poly(A, R, v)
    A.vals[A.nnz // 2] += 0.25
    A.vals[7] = float("inf")
    ref = _csr_steps(p, torch, A, R, v)
    got = p.apply_poly(A, R, v)
    assert torch.equal(torch.nan_to_num(got), torch.nan_to_num(ref))
    assert torch.equal(torch.isfinite(got), torch.isfinite(ref))
