"""The solve on one thread-block cluster (systems with narrow levels) at the sizes
where it can go wrong: systems shorter than a window, windows that end inside a
level and inside a chain, one row past a window, rows longer than the entries a warp
holds, upper and transposed systems, and values that never come.  The level-order
tiles fold every row in the same order at the same width, so results must be
bitwise equal to theirs."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import TOL64, dev, long_rows, plan_for, relerr, unit_without_diagonal

pytestmark = pytest.mark.gpu

WINDOW = {torch.float64: 12288, torch.float32: 24576}   # rows


@pytest.fixture(scope="module", autouse=True)
def _gpu(cuda_device):
    yield


def _chains(n, width, upper=False):
    """`width` interleaved chains: row i needs row i - width."""
    i = np.arange(n)
    far = i[width:]
    r = np.concatenate([i, far])
    c = np.concatenate([i, far - width])
    if upper:
        r, c = n - 1 - r, n - 1 - c
    order = np.lexsort((c, r))
    r, c = r[order], c[order]
    return synth._from_sorted_coo(n, r, c, np.where(r == c, 2.0, -1.0), upper=upper)


def _irregular(n, upper=False, seed=5):
    """0 to 40 dependencies a row, most of them on the last 64 rows."""
    rng = np.random.default_rng(seed)
    r, c = [], []
    for i in range(n):
        k = min(i, int(rng.integers(0, 41)) if i % 7 == 0 else int(rng.integers(1, 9)))
        near = i - 1 - rng.integers(0, min(i, 64), k) if i else np.zeros(0, int)
        far = rng.integers(0, i, k) if i else np.zeros(0, int)
        cols = np.unique(np.append(np.where(rng.random(k) < 0.8, near, far), i))
        r.append(np.full(cols.size, i))
        c.append(cols)
    r, c = np.concatenate(r), np.concatenate(c)
    if upper:
        r, c = (n - 1 - r)[::-1], (n - 1 - c)[::-1]
    return synth._from_sorted_coo(n, r, c, np.where(r == c, 60.0, -1.0), upper=upper)


MATRICES = {
    "chain_one_window": lambda h: _chains(h, 1),
    "chain_one_row_more": lambda h: _chains(h + 1, 1),
    "chains_5": lambda h: _chains(2 * h + 77, 5),
    "chains_5_upper": lambda h: _chains(2 * h + 77, 5, upper=True),
    "irregular_short": lambda h: _irregular(997),
    "irregular": lambda h: _irregular(3 * h - 5),
    "irregular_upper": lambda h: _irregular(h + 31, upper=True),
    "long_rows": lambda h: long_rows(),
    "unit_nodiag": lambda h: unit_without_diagonal(),
}


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("name", sorted(MATRICES))
def test_every_width_is_bitwise_the_tiled_form(name, dtype):
    A = MATRICES[name](WINDOW[dtype])
    b = torch.tensor(synth.uniform(A.n, 41), device=dev(), dtype=dtype)
    with plan_for(A, dtype=dtype) as p:
        for lanes in (16, 32):
            p.set_tuning(lanes, 256, 0)
            for solve in (p.solve, p.solve_transpose):
                want = solve(b, algo="blocked")
                for algo in ("self", "permuted"):
                    assert torch.equal(solve(b, algo=algo), want), (lanes, algo)
                    x = b.clone()
                    assert torch.equal(solve(x, out=x, algo=algo), want), (lanes, algo)
        assert p.status() == (0, -1)
        if dtype == torch.float64:
            ref = oracle.solve(A.rowptr, A.colidx, A.vals, b.cpu().numpy(), upper=A.upper,
                               unit=A.unit)
            assert relerr(p.solve(b), ref) <= TOL64


@pytest.mark.parametrize("algo", ["self", "permuted"])
@pytest.mark.parametrize("lanes", [16, 32])
def test_a_value_that_never_comes_holds_up_only_its_dependents(lanes, algo):
    """Seven chains through four windows, one row of the first withheld."""
    width, held = 7, 5003
    A = _chains(3 * WINDOW[torch.float64] + 501, width)
    b = synth.uniform(A.n, 43)
    ref = oracle.solve(A.rowptr, A.colidx, A.vals, b)
    i = np.arange(A.n)
    behind = (i > held) & (i % width == held % width)
    free = ~behind & (i != held)
    with plan_for(A) as p:
        p.set_tuning(lanes, 256, 0)
        p.set_spin_limit(1 << 12)
        p.withhold_row(held)
        got = p.solve(torch.tensor(b, device=dev()), algo=algo).cpu().numpy()
        assert p.last_launch_count == 1
        assert p.status() == (6, held + width)
        assert np.all(np.isnan(got[behind]))
        assert relerr(got[free], ref[free]) <= TOL64
        p.withhold_row(-1)
        p.set_spin_limit(1)      # every wait runs out: level by level, still exact
        x = torch.tensor(b, device=dev())
        assert relerr(p.solve(x, out=x, algo=algo), ref) <= TOL64
        assert p.status() == (0, -1)
