"""GPU: the forms of a chain and of an Arnoldi step are the ones taken.  Each
has another to fall back on with the same results, so results do not show it."""
import numpy as np
import pytest

import synth
from gpu_util import dev_csr, ppg_or_skip, to_dev
from test_gpu_diagonals import CASES, GRID, _banded

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
