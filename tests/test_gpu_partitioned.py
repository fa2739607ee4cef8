"""The sliced copy and the kernel of the partitioned solve at the sizes where
they can go wrong: rows longer than the chunks a warp loads ahead, in the part
and out of it, empty rows, parts of one row, copies that would be mostly
padding, and values that never come.  The in-place form folds every row in the
same order at the same width, so results must be bitwise equal to its."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import (TOL64, bidiagonal, dev, diagonal, long_rows, plan_for, relerr,
                      unit_without_diagonal)

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu(cuda_device):
    yield


def _band(n, width):
    """Every row i holds columns i - width .. i: `width` entries per row in and,
    for small parts, out of the part."""
    i = np.repeat(np.arange(n), width + 1)
    j = i - np.tile(np.arange(width, -1, -1), n)
    keep = j >= 0
    i, j = i[keep], j[keep]
    return synth._from_sorted_coo(n, i, j, np.where(i == j, 2.0 * width, -1.0), upper=False)


MATRICES = {
    "band_1": lambda: bidiagonal(700),
    "band_7": lambda: _band(900, 7),
    "band_64": lambda: _band(700, 64),
    "diagonal": lambda: diagonal(515),
    "long_rows": lambda: long_rows(),
    "unit_nodiag": lambda: unit_without_diagonal(),
    "grid27_upper": lambda: synth.laplacian_triangles((13, 7, 9), 27)[1],
    "one_row": lambda: diagonal(1),
}


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("name", sorted(MATRICES))
def test_every_width_and_part_size_is_bitwise_the_in_place_form(name, dtype):
    A = MATRICES[name]()
    b = torch.tensor(synth.uniform(A.n, 61), device=dev(), dtype=dtype)
    with plan_for(A, dtype=dtype) as p:
        for lanes in (1, 2, 8, 32):
            for block in (32, 512, 1024):
                p.set_tuning(lanes, block, 0)
                want = p.solve(b, algo="self")
                want_t = p.solve_transpose(b, algo="self")
                for rows, cl in ((1, 1), (37, 1), (64, 4), (0, 2), (1 << 30, 1)):
                    p.set_partition(rows, cl)
                    assert torch.equal(p.solve(b, algo="partitioned"), want), (lanes, rows, cl)
                assert torch.equal(p.solve_transpose(b, algo="partitioned"), want_t)
        assert p.status() == (0, -1)


def test_mostly_padding_runs_on_the_level_ordered_copy():
    """Every 32nd row holds 60 entries, the others only their diagonal: at one
    lane per row a slice would hold one entry in 32 slots."""
    n = 100_000
    lens = np.where((np.arange(n) % 32 == 31) & (np.arange(n) >= 64), 60, 1)
    i = np.repeat(np.arange(n), lens)
    k = np.arange(i.size) - np.repeat(np.cumsum(lens) - lens, lens)
    j = i - (np.repeat(lens, lens) - 1 - k)
    A = synth._from_sorted_coo(n, i, j, np.where(i == j, 60.0, -1.0), upper=False)
    b = torch.tensor(synth.uniform(n, 67), device=dev())
    with plan_for(A) as p:
        p.set_tuning(1, 256, 0)
        want = p.solve(b, algo="self")
        assert torch.equal(p.solve(b, algo="partitioned"), want)
        p.prepare("partitioned")
        g = torch.cuda.CUDAGraph()
        x = torch.empty_like(b)
        with torch.cuda.graph(g):
            p.solve(b, out=x, algo="partitioned")
        g.replay()
        assert torch.equal(x, want)
        vals = 2.0 * p.vals          # new values reach the copy that is used
        p.set_values(vals)
        assert torch.equal(p.solve(b, algo="partitioned"), p.solve(b, algo="self"))
        x, _, _ = p.solve_refined(b)
        assert relerr(x, oracle.solve(A.rowptr, A.colidx, 2.0 * A.vals, b.cpu().numpy())) <= TOL64


@pytest.mark.parametrize("cluster", [1, 2])
@pytest.mark.parametrize("lanes", [1, 4])
def test_a_value_that_never_comes_holds_up_only_its_dependents(lanes, cluster):
    """5-point grid with one row withheld: every row that does not depend on it
    is exact although warps hold groups that do, the first dependent row is
    reported, and the next solve is clean."""
    nx, ny = 40, 33
    A = synth.lap2d_5pt_lower(nx, ny)
    held = 7 * nx + 11
    x, y = np.arange(A.n) % nx, np.arange(A.n) // nx
    below = (x >= held % nx) & (y >= held // nx)     # depends on the withheld row
    below[held] = False
    b = synth.uniform(A.n, 71)
    ref = oracle.solve(A.rowptr, A.colidx, A.vals, b)
    with plan_for(A) as p:
        p.set_tuning(lanes, 64, 0)
        p.set_partition(3 * nx, cluster)
        p.set_spin_limit(1 << 14)
        p.withhold_row(held)
        got = p.solve(torch.tensor(b, device=dev()), algo="partitioned").cpu().numpy()
        free = ~below
        free[held] = False
        assert p.status() == (6, held + 1)
        assert np.all(np.isnan(got[below]))
        assert relerr(got[free], ref[free]) <= TOL64
        p.withhold_row(-1)
        assert relerr(p.solve(torch.tensor(b, device=dev()), algo="partitioned"), ref) <= TOL64
        assert p.status() == (0, -1)


@pytest.mark.parametrize("in_place", [False, True])
def test_capture_at_a_width_that_was_not_prepared(in_place):
    """A captured solve cannot build the copy of another width: it runs on what is
    there, also in place, with the result of that width."""
    A = synth.laplacian_triangles((13, 17, 9), 7)[0]
    b = torch.tensor(synth.uniform(A.n, 73), device=dev())
    with plan_for(A) as p:
        p.set_tuning(1, 128, 0)
        p.prepare("partitioned")
        p.set_tuning(4, 128, 0)
        x = b.clone() if in_place else torch.empty_like(b)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            p.solve(x if in_place else b, out=x, algo="partitioned")
        g.replay()
        assert torch.equal(x, p.solve(b, algo="self"))
        assert torch.equal(x, p.solve(b, algo="partitioned"))
        assert p.status() == (0, -1)
