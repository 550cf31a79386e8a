"""GPU: long rows in the kernels that stage a matrix streamed from memory, against
the small matrix's direct steps, bit for bit."""
import numpy as np
import pytest

from gpu_util import dev_csr, ppg_or_skip, random_csr, to_dev

pytestmark = pytest.mark.gpu

# tiles are 128 rows in FP64 and 512 in FP32, where a thread owns rows t and t + 256;
# a chunk is 1,024 entries in FP64, 3,584 (with long rows 3,040) in FP32
HEADS = {
    # both rows of one thread, rows over several chunks, all of a warp's rows, the
    # last row of a tile and of the head
    "few": dict(n=3001, long_rows={0: 129, 10: 400, 266: 700, 300: 2900, 511: 200, 512: 130, 700: 1100,
                                   3000: 333}, empty_rows={1, 36, 2000}),
    "a_warp": dict(n=2500, long_rows={**{r: 129 + r % 40 for r in range(96, 130)}, 1500: 2400}),
    "every_fourth": dict(n=2600, long_rows={r: 140 for r in range(0, 2600, 4)}),
    "most": dict(n=1100, long_rows={r: 120 + r % 200 for r in range(0, 1100)}),
}
ROOTS = np.array([4.0, 3 + 1j, 3 - 1j, 2.5, 2 + 0.5j, 2 - 0.5j, 3.3], dtype=complex)
LONG_ROOTS = np.array([4.0 + 0.02 * k for k in range(24)])


@pytest.fixture(scope="module")
def env():
    return ppg_or_skip()


def _streamed(p, torch, A, per_row, nnz=1.5e7):
    """A as the head of a block-diagonal matrix too large for L2: rows of per_row
    entries on and behind the diagonal, which go round at the end."""
    n = int(nnz / per_row)
    row = torch.arange(n, device="cuda").repeat_interleave(per_row)
    col = (row + torch.arange(per_row, device="cuda").repeat(n)) % n
    col = col.view(n, per_row).sort(1).values.reshape(-1)
    rp = torch.arange(1, n + 1, device="cuda") * per_row + A.nnz
    return p.CSR(torch.cat([A.rowptr, rp.int()]), torch.cat([A.colind, (col + A.n).int()]),
                 torch.cat([A.vals, torch.full((col.numel(),), 2.0 / per_row, dtype=A.dtype, device="cuda")]))


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("per_row", [5, 20, 150])   # in FP32: read twice, from the chunks, all tiles long
@pytest.mark.parametrize("name", sorted(HEADS))
def test_staged_equals_direct(env, name, per_row, dtype):
    p, torch = env
    tdt = torch.float64 if dtype == "f64" else torch.float32
    A = dev_csr(p, torch, random_csr(seed=3, **HEADS[name]), dtype=tdt)
    big = _streamed(p, torch, A, per_row)
    assert p.chain_form(A, 1) == "direct"
    assert p.chain_form(big, 7) == "staged" and p.chain_form(big, 30) == "staged"
    v = to_dev(torch, np.random.default_rng(9).standard_normal(A.n), tdt)
    vb = torch.cat([v, torch.ones(big.n - A.n, dtype=tdt, device="cuda")])
    assert torch.equal(p.spmv(big, vb)[: A.n], p.spmv(A, v))
    for roots in (ROOTS, LONG_ROOTS):   # (24 steps: FP32 looks for diagonals)
        R = p.Roots.from_complex(roots)
        assert torch.equal(p.apply_poly(big, R, vb)[: A.n], p.apply_poly(A, R, v))
        assert torch.equal(p.apply_phi(big, R, vb)[: A.n], p.apply_phi(A, R, v))


@pytest.mark.parametrize("name", ["every_fourth", "most"])
def test_rows_over_chunk_ends_many_times(env, name):
    """Every chunk ends within a long row and begins within another's rest, which
    two warps have at the same time."""
    p, torch = env
    A = dev_csr(p, torch, random_csr(seed=3, **HEADS[name]), dtype=torch.float32)
    v = to_dev(torch, np.random.default_rng(9).standard_normal(A.n), torch.float32)
    k = 60
    off = torch.arange(k, device="cuda").repeat_interleave(A.nnz)
    rp = torch.cat([A.rowptr[:-1].long().repeat(k) + torch.arange(k, device="cuda").repeat_interleave(A.n) * A.nnz,
                    torch.tensor([k * A.nnz], device="cuda")])
    copies = p.CSR(rp.int(), (A.colind.long().repeat(k) + off * A.n).int(), A.vals.repeat(k))
    big = _streamed(p, torch, copies, 20)
    R = p.Roots.from_complex(ROOTS)
    ref = p.apply_phi(A, R, v).repeat(k)
    vb = torch.cat([v.repeat(k), torch.ones(big.n - copies.n, dtype=torch.float32, device="cuda")])
    assert p.chain_form(big, 7) == "staged"
    for _ in range(20):
        assert torch.equal(p.apply_phi(big, R, vb)[: copies.n], ref)


@pytest.mark.parametrize("per_row", [5, 150])
def test_residual_with_long_rows(env, per_row):
    """The residual's norm: one cycle of one step from x0, against the residual
    vector's (summed in another order: a few units of the last place)."""
    p, torch = env
    A = dev_csr(p, torch, random_csr(seed=3, **HEADS["few"]))
    big = _streamed(p, torch, A, per_row)
    x0 = torch.ones(big.n, dtype=torch.float64, device="cuda")
    b = to_dev(torch, np.random.default_rng(8).standard_normal(big.n))
    x, st = p.solve(big, b, m=1, tol=1e-30, x0=x0, max_cycles=1)
    r = b - p.spmv(big, x)
    assert abs(st["true_relres"] - float(r.norm() / b.norm())) <= 1e-13 * st["true_relres"]


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("n", [200, 1101, 1102, 1103, 32768])
def test_few_rows_to_a_warp(env, n, dtype):
    """More than 22 entries in the average row of a small system: four rows to a
    warp, the last one with fewer, short and long."""
    p, torch = env
    tdt = torch.float64 if dtype == "f64" else torch.float32
    lens = {r: 129 + r % 90 for r in range(0, n, 5)} if n < 5000 else {r: 400 for r in range(0, n, 16)}
    A = dev_csr(p, torch, random_csr(n, 6, long_rows=lens, empty_rows={1}), dtype=tdt)
    assert A.nnz > 22 * n
    big = _streamed(p, torch, A, 5)
    v = to_dev(torch, np.random.default_rng(9).standard_normal(A.n), tdt)
    vb = torch.cat([v, torch.ones(big.n - A.n, dtype=tdt, device="cuda")])
    assert p.chain_form(A, 7) == "direct" and p.chain_form(big, 7) == "staged"
    assert torch.equal(p.spmv(big, vb)[: A.n], p.spmv(A, v))
    R = p.Roots.from_complex(ROOTS)
    assert torch.equal(p.apply_poly(big, R, vb)[: A.n], p.apply_poly(A, R, v))
    assert torch.equal(p.apply_phi(big, R, vb)[: A.n], p.apply_phi(A, R, v))
