"""GPU: the forms of a chain and of an Arnoldi step are the ones taken.  Each
has another to fall back on with the same results, so results do not show it."""
import os
import subprocess
import sys

import numpy as np
import pytest

import synth
from gpu_util import dev_csr, ppg_or_skip, to_dev
from test_gpu_diagonals import CASES, GRID, _banded, _csr_steps, _roots

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    return ppg_or_skip()


@pytest.mark.parametrize("name,form", [
    ("one_value_each", "diagonals_2"),
    ("an_even_number_of_tiles", "diagonals_2"),
    ("some_own_values", "diagonals_2"),
    ("dropped_entries", "diagonals"),
    ("close_offsets", "diagonals"),
    ("nine", "diagonals"),
    ("forty", "staged"),
])
def test_diagonal_form(env, name, form):
    p, torch = env
    A = dev_csr(p, torch, _banded(**CASES[name]), dtype=torch.float32)
    assert p.chain_form(A, 33) == form
    assert p.chain_form(A, 3) == "staged"          # not repaid
    assert p.chain_form(A.astype(torch.float64), 33) == "staged"


def test_unsorted_row_has_no_diagonal_form(env):
    p, torch = env
    H = _banded(GRID)
    k = H.rowptr[400_000]
    H.colind[[k, k + 1]] = H.colind[[k + 1, k]]
    A = p.CSR.from_host(H.rowptr, H.colind, H.vals, dtype=torch.float32, validate=False)
    assert p.chain_form(A, 33) == "staged"


OFF27 = [i * 10000 + j * 100 + k for i in (-1, 0, 1) for j in (-1, 0, 1) for k in (-1, 0, 1)]


@pytest.mark.parametrize("name,kw,form", [
    # more entries to a tile of the search than it holds at once
    ("twenty_seven_of_one_value", dict(offsets=OFF27, one_value=OFF27, n=1_300_001), "diagonals"),
    # more values of their own than a tile's shared memory holds
    ("thirteen_apart", CASES["thirteen_apart"], "staged"),
    ("twenty_seven_own", dict(offsets=OFF27, n=1_300_001), "staged"),
    # the middle row, which the list starts from, and the tiles' first rows empty
    ("empty_rows", dict(offsets=GRID, drop=0.2, empty=[1_300_001] + list(range(0, 2_600_000, 128))),
     "diagonals"),
])
def test_search_for_the_diagonals(env, name, kw, form):
    """... and p(A) v over the form found equals the CSR steps."""
    p, torch = env
    A = dev_csr(p, torch, _banded(**kw), dtype=torch.float32)
    assert p.chain_form(A, 33) == form
    v = to_dev(torch, np.random.default_rng(4).standard_normal(A.n), torch.float32)
    R = p.Roots.from_complex(_roots())
    assert torch.equal(p.apply_poly(A, R, v), _csr_steps(p, torch, A, R, v))


def test_an_offset_late_in_the_matrix(env):
    """Rows with an offset of their own near the end: one more diagonal, or (forty
    of them) no form; and single entries whose value differs."""
    p, torch = env
    R = p.Roots.from_complex(_roots())
    v = to_dev(torch, np.random.default_rng(4).standard_normal(2_600_003), torch.float32)
    for rows, form in ((1, "diagonals_2"), (40, "staged")):
        H = _banded(GRID, one_value=GRID)
        for r in range(2_500_000, 2_500_000 + rows):
            H.colind[H.rowptr[r + 1] - 1] = 2_510_000
        H.vals[[5, H.rowptr[2_599_000]]] = 0.125
        A = dev_csr(p, torch, H, dtype=torch.float32)
        assert p.chain_form(A, 33) == form
        assert torch.equal(p.apply_poly(A, R, v), _csr_steps(p, torch, A, R, v))


def test_small_and_l2_held_systems(env):
    p, torch = env
    for dtype in (torch.float64, torch.float32):
        small = dev_csr(p, torch, synth.cd2d(50, 0.5), dtype=dtype)
        assert p.chain_form(small, 10) == "cluster"
        assert p.chain_form(small, 1) == "direct"
        assert p.chain_form(dev_csr(p, torch, synth.cd2d(300, 0.5), dtype=dtype), 40) == "direct"


def test_launches_of_a_small_system(env):
    p, torch = env
    A = dev_csr(p, torch, synth.cd2d(50, 0.5))
    v = to_dev(torch, np.random.default_rng(1).standard_normal(A.n))
    R = p.Roots.from_complex(np.array([5 + 2j, 5 - 2j] * 5))
    before = p.lib.ppg_launch_count()
    p.apply_poly(A, R, v)
    assert p.lib.ppg_launch_count() - before == 1
    # an Arnoldi step: the product and the orthogonalisation (six launches more
    # one by one), and a few launches around the cycle
    _, st = p.solve(A, v, m=20, tol=1e-30, max_cycles=1)
    assert st["launches"] <= 2 * 20 + 12
    before = p.lib.ppg_launch_count()
    p.build_poly(A, 20, v)
    assert p.lib.ppg_launch_count() - before <= 2 * 20 + 12


def test_chain_statistics_of_a_small_system(env):
    """A chain in one launch counts as one, with the matrix read once."""
    p, torch = env
    H = synth.cd2d(50, 0.5)
    A = dev_csr(p, torch, H)
    b = to_dev(torch, np.random.default_rng(1).standard_normal(A.n))
    R = p.build_poly(A, 10, b)
    _, st = p.solve(A, b, m=20, tol=1e-8, roots=R, timing=True)
    chains = st["iters"] + st["cycles"]
    assert st["poly_launches"] == chains and st["poly_launches"] < st["launches"]
    csr = 12 * H.rowptr[-1] + 4 * (H.n + 1)
    assert st["poly_bytes"] == st["iters"] * (csr + 16 * H.n) + st["cycles"] * (csr + 24 * H.n)
    assert 0 < st["poly_ms"]


def test_chain_statistics_by_diagonals(env):
    """A grid's FP32 steps by its diagonals, all of one value: a byte of mask to a row
    and two to four vectors; and by the CSR without the form."""
    p, torch = env
    for name, kw in (("grid", CASES["one_value_each"]), ("none", CASES["forty"])):
        H = _banded(**kw)
        A = dev_csr(p, torch, H)
        b = to_dev(torch, np.random.default_rng(1).standard_normal(A.n))
        R = p.Roots.from_complex(_roots())
        _, st = p.solve_flex(A, A.astype(torch.float32), b, R, m=2, tol=1e-30, max_cycles=1, timing=True)
        per_row = st["poly_bytes"] / st["poly_launches"] / A.n
        csr = 8 * H.rowptr[-1] / H.n
        assert (1 + 8 <= per_row <= 1 + 16) if name == "grid" else (csr + 8 <= per_row <= csr + 4 + 16.1)
        assert st["poly_launches"] == 2 * 33


def test_no_room_for_the_diagonal_form(env):
    """In a process of its own, whose other allocator holds all but 1.5 GB: the form's
    250 MB stay untaken, and the result is that of the CSR steps."""
    code = """
import sys
sys.path.insert(0, "tests")
import numpy as np, torch, paper_1911_07065_gb300 as p
from test_gpu_diagonals import GRID, _banded, _roots
H = _banded(GRID, n=5_000_000)
A = p.CSR.from_host(H.rowptr, H.colind, H.vals, dtype=torch.float32)
v = torch.ones(A.n, dtype=torch.float32, device="cuda")
R = p.Roots.from_complex(_roots())
torch.cuda.synchronize()
held = torch.empty(torch.cuda.mem_get_info()[0] - 1500 * 2**20, dtype=torch.uint8, device="cuda")
assert p.chain_form(A, 33) == "staged"
y = p.apply_poly(A, R, v)
torch.cuda.synchronize()
assert torch.cuda.mem_get_info()[0] > 1300 * 2**20
del held
torch.cuda.empty_cache()
assert p.chain_form(A, 33) == "diagonals"
assert torch.equal(p.apply_poly(A, R, v), y)
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    subprocess.run([sys.executable, "-c", code], check=True, cwd=root, timeout=300)


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("n", [300, 4000, 9000, 16384])
def test_rows_beyond_the_registers_in_one_cluster(env, n, dtype):
    """Rows of nine to some hundred entries among short ones, one and (above 8,192 rows,
    FP32) two rows to a thread, against the same rows step by step."""
    p, torch = env
    tdt = torch.float64 if dtype == "f64" else torch.float32
    if dtype == "f64" and n > 9000:
        pytest.skip("more multiply-adds than the FP64 cluster takes")
    lens = np.where(np.arange(n) % 97 == 5, 90, np.where(np.arange(n) % 31 == 7, 9 + np.arange(n) % 12, 3))
    lens[[0, n - 1]] = 30, 140
    rng = np.random.default_rng(3)
    cols = [np.unique(np.concatenate([rng.integers(0, n, k - 1), [i]])) for i, k in enumerate(lens)]
    rowptr = np.concatenate([[0], np.cumsum([c.size for c in cols])]).astype(np.int32)
    H = synth.CSRHost(n, rowptr, np.concatenate(cols).astype(np.int32), 0.1 * rng.standard_normal(rowptr[-1]))
    A = dev_csr(p, torch, H, dtype=tdt)
    extra = 40000 - n
    big = p.CSR(torch.cat([A.rowptr, A.nnz + torch.arange(1, extra + 1, dtype=torch.int32, device="cuda")]),
                torch.cat([A.colind, A.n + torch.arange(extra, dtype=torch.int32, device="cuda")]),
                torch.cat([A.vals, torch.full((extra,), 5.0, dtype=tdt, device="cuda")]))
    assert p.chain_form(A, 33) == "cluster" and p.chain_form(big, 33) == "direct"
    v = to_dev(torch, rng.standard_normal(n), tdt)
    vb = torch.cat([v, torch.ones(extra, dtype=tdt, device="cuda")])
    R = p.Roots.from_complex(_roots())
    assert torch.equal(p.apply_poly(A, R, v), p.apply_poly(big, R, vb)[:n])
    assert torch.equal(p.apply_phi(A, R, v), p.apply_phi(big, R, vb)[:n])
