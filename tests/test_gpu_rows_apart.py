"""The kernel that takes every row at its own pace, on the systems that reach it: rows
that differ at few lanes, one lane per row, levels of very many rows; and values that
never come, with so few warps that they own every ticket.  The blocked form folds every
row in the same order at the same width, so results must be bitwise its."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import TOL64, bidiagonal, dev, diagonal, long_rows, plan_for, relerr, \
    unit_without_diagonal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu(cuda_device):
    yield


def _two_levels(n, k, upper=False, seed=3):
    """Rows past n / 2 need up to k random rows of the first half."""
    rng = np.random.default_rng(seed)
    i, h = np.arange(n), n // 2
    r = np.repeat(np.arange(h, n), k)
    key = np.unique(np.concatenate([i * n + i, r.astype(np.int64) * n + rng.integers(0, h, r.size)]))
    r, c = key // n, key % n
    if upper:
        r, c = (n - 1 - r)[::-1], (n - 1 - c)[::-1]
    return synth._from_sorted_coo(n, r, c, np.where(r == c, 4.0 * k, -1.0), upper=upper)


MATRICES = {
    "chain": lambda: bidiagonal(2100),
    "chain_upper": lambda: bidiagonal(2100, upper=True),
    "long_rows": lambda: long_rows(3001),
    "unit_nodiag": lambda: unit_without_diagonal(2000),
    "grid5": lambda: synth.lap2d_5pt_lower(130, 131),          # one lane per row
    "diagonal": lambda: diagonal(600_001),                     # over 8192 tickets a level
    "two_levels": lambda: _two_levels(600_003, 5),
    "two_levels_upper": lambda: _two_levels(600_003, 5, upper=True),
}


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("name", sorted(MATRICES))
def test_every_width_is_bitwise_the_blocked_form(name, dtype):
    A = MATRICES[name]()
    b = torch.tensor(synth.uniform(A.n, 51), device=dev(), dtype=dtype)
    with plan_for(A, dtype=dtype) as p:
        for lanes in (1, 2, 4, 8, 16, 32):
            for block, cap in ((64, 3), (256, 304), (1024, 0)):
                p.set_tuning(lanes, block, cap)
                for solve in (p.solve, p.solve_transpose):
                    want = solve(b, algo="blocked")
                    for algo in ("self", "permuted"):
                        assert torch.equal(solve(b, algo=algo), want), (lanes, block, algo)
                        x = b.clone()
                        assert torch.equal(solve(x, out=x, algo=algo), want), (lanes, block, algo)
        assert p.status() == (0, -1)
        if dtype == torch.float64:
            ref = oracle.solve(A.rowptr, A.colidx, A.vals, b.cpu().numpy(), upper=A.upper,
                               unit=A.unit)
            assert relerr(p.solve(b), ref) <= TOL64


@pytest.mark.parametrize("algo", ["self", "permuted"])
@pytest.mark.parametrize("lanes", [1, 2, 4])
def test_a_withheld_row_holds_up_only_its_dependents(lanes, algo):
    A = synth.block_diagonal([synth.general_lower(900, 5), synth.general_lower(2500, 6)])
    held = 500
    behind = np.zeros(A.n, dtype=bool)
    behind[held] = True
    for i in range(held + 1, A.n):
        behind[i] = behind[A.colidx[A.rowptr[i]:A.rowptr[i + 1] - 1]].any()
    free = ~behind
    behind[held] = False
    b = synth.uniform(A.n, 53)
    ref = oracle.solve(A.rowptr, A.colidx, A.vals, b)
    with plan_for(A) as p:
        p.set_tuning(lanes, 64, 1)
        p.set_spin_limit(1 << 12)
        p.withhold_row(held)
        got = p.solve(torch.tensor(b, device=dev()), algo=algo).cpu().numpy()
        assert p.status() == (6, int(np.flatnonzero(behind)[0]))
        assert np.all(np.isnan(got[behind]))
        assert relerr(got[free], ref[free]) <= TOL64
        p.withhold_row(-1)
        assert relerr(p.solve(torch.tensor(b, device=dev()), algo=algo), ref) <= TOL64
        assert p.status() == (0, -1)
