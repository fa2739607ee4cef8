"""The solve on one thread-block cluster where a window ends: systems of exactly one and
two windows, one row more, windows that end inside a level.  One row and one column are
long, so that neither direction has like rows: such a system runs in one launch only on
the cluster (the one-block kernel wants like rows, every other form has two launches)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import TOL64, dev, plan_for, relerr

pytestmark = pytest.mark.gpu

WINDOW = {torch.float64: 12288, torch.float32: 24576}   # rows


@pytest.fixture(scope="module", autouse=True)
def _gpu(cuda_device):
    yield


def _chains(n, width, upper=False):
    """`width` interleaved chains; the last row needs 300 rows more, 300 rows need row 0."""
    rng = np.random.default_rng(n)
    i = np.arange(n)
    far = i[width:]
    r = np.concatenate([i, far, np.full(300, n - 1), rng.choice(n - 2, 300, replace=False) + 1])
    c = np.concatenate([i, far - width, rng.choice(n - 1, 300, replace=False), np.zeros(300, int)])
    if upper:
        r, c = n - 1 - r, n - 1 - c
    key = np.unique(r.astype(np.int64) * n + c)
    r, c = key // n, key % n
    return synth._from_sorted_coo(n, r, c, np.where(r == c, 400.0, -1.0), upper=upper)


def _unlike(A):
    rows, cols = np.diff(A.rowptr), np.bincount(A.colidx, minlength=A.n)
    return min(rows.max(), cols.max()) * A.n > 2 * A.nnz + 2 * A.n


SHAPES = {
    "one_window": lambda h: (h, 1, False),
    "one_row_more": lambda h: (h + 1, 1, False),
    "two_windows": lambda h: (2 * h, 3, False),
    "two_windows_one_row_more": lambda h: (2 * h + 1, 5, True),
    "ends_inside_a_level": lambda h: (2 * h + 77, 7, True),
}


@pytest.mark.parametrize("lanes", [16, 32])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("name", sorted(SHAPES))
def test_both_forms_and_directions_also_captured(name, dtype, lanes):
    A = _chains(*SHAPES[name](WINDOW[dtype]))
    assert _unlike(A)
    b = torch.tensor(synth.uniform(A.n, 43), device=dev(), dtype=dtype)
    with plan_for(A, dtype=dtype) as p:
        p.set_tuning(lanes, 256, 0)
        for solve in (p.solve, p.solve_transpose):
            want = solve(b, algo="blocked")
            for algo in ("self", "permuted"):
                assert torch.equal(solve(b, algo=algo), want), algo
                assert p.last_launch_count == 1, algo
                x = b.clone()
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g):
                    solve(x, out=x, algo=algo)
                g.replay()
                assert torch.equal(x, want), algo
                x.copy_(b)
                g.replay()
                assert torch.equal(x, want), algo
        assert p.status() == (0, -1)
        if dtype == torch.float64:
            ref = oracle.solve(A.rowptr, A.colidx, A.vals, b.cpu().numpy(), upper=A.upper)
            assert relerr(p.solve(b), ref) <= TOL64


@pytest.mark.parametrize("algo", ["self", "permuted"])
@pytest.mark.parametrize("extra", [0, 1])
def test_fp32_steps_of_a_refined_solve(extra, algo):
    A = _chains(WINDOW[torch.float32] + extra, 3)
    b = torch.tensor(synth.uniform(A.n, 47), device=dev())
    with plan_for(A) as p:
        p.set_tuning(32, 256, 0)
        got = []
        for form in ("blocked", algo):
            p.best_algo = form
            got.append(p.solve_refined(b)[0])
        assert torch.equal(got[0], got[1])
        assert relerr(got[1], oracle.solve(A.rowptr, A.colidx, A.vals, b.cpu().numpy())) <= TOL64
        assert p.status() == (0, -1)
