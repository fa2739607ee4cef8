"""The two ways in which the self-scheduled kernel takes a ticket's rows, and the
solve in one block, at their edges: rows of one and of several chunks, tickets
that straddle levels, systems just inside and outside shared memory.  All are
compared with the oracle, and with each other where the order of a row's sums is
the same (equal lanes per row)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import TOL32, TOL64, bidiagonal, dev, diagonal, plan_for, relerr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu(cuda_device):
    yield


def _band(n, width, every=1):
    """Row i holds columns i - width .. i, but only itself unless i is a multiple
    of `every`."""
    w = np.where(np.arange(n) % every == 0, width, 0)
    w = np.minimum(w, np.arange(n))
    i = np.repeat(np.arange(n), w + 1)
    j = i - (np.repeat(np.cumsum(w + 1), w + 1) - 1 - np.arange(i.size))
    return synth._from_sorted_coo(n, i, j, np.where(i == j, 2.0 * width, -1.0), upper=False)


MATRICES = {
    # alike, narrow: one block
    "grid5_30x41": lambda: synth.lap2d_5pt_lower(30, 41),
    "grid5_upper": lambda: synth.lap2d_5pt_upper(33, 9),
    # alike, the largest FP64 systems of one block (shared memory) and one row more
    "grid5_fits": lambda: synth.lap2d_5pt_lower(44, 660),
    "grid5_too_large": lambda: synth.lap2d_5pt_lower(44, 661),
    # alike, wide levels, several chunks at few lanes
    "grid27": lambda: synth.laplacian_triangles((17, 13, 11), 27)[0],
    # one row per level
    "chain": lambda: bidiagonal(1500),
    "band_40": lambda: _band(800, 40),
    # long rows among short ones
    "band_40_every_5": lambda: _band(900, 40, 5),
    "general": lambda: synth.general_lower(4000, 77),
    "diagonal": lambda: diagonal(33),
}


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("name", sorted(MATRICES))
def test_in_place_and_copy_forms_at_every_width(name, dtype):
    A = MATRICES[name]()
    b = synth.uniform(A.n, 81)
    tol = TOL64 if dtype == torch.float64 else TOL32
    ref = oracle.solve(A.rowptr, A.colidx, A.vals, b, upper=A.upper)
    ref_t = oracle.solve_transpose(A.rowptr, A.colidx, A.vals, b, upper=A.upper)
    bt = torch.tensor(b, device=dev(), dtype=dtype)
    with plan_for(A, dtype=dtype) as p:
        for lanes in (1, 2, 4, 8, 16, 32):
            for block, cap in ((32, 1), (256, 0), (1024, 2)):
                p.set_tuning(lanes, block, cap)
                x = p.solve(bt, algo="self")
                assert relerr(x.double(), ref) <= tol, (lanes, block)
                assert torch.equal(p.solve(bt, algo="permuted"), x), (lanes, block)
                # the blocked form keeps its own kernel: same order, same bits
                assert torch.equal(p.solve(bt, algo="blocked"), x), (lanes, block)
                inplace = bt.clone()
                assert torch.equal(p.solve(inplace, out=inplace, algo="self"), x)
                inplace = bt.clone()
                assert torch.equal(p.solve(inplace, out=inplace, algo="permuted"), x)
            assert relerr(p.solve_transpose(bt).double(), ref_t) <= tol
        assert p.status() == (0, -1)


@pytest.mark.parametrize("shape", [(24, 31), (60, 700)])
def test_a_withheld_row_holds_up_only_its_dependents(shape):
    """In one block and on the whole GPU: rows that do not depend on the
    withheld row are exact although their tickets hold rows that do."""
    nx, ny = shape
    A = synth.lap2d_5pt_lower(nx, ny)
    held = 5 * nx + 7
    x, y = np.arange(A.n) % nx, np.arange(A.n) // nx
    below = (x >= held % nx) & (y >= held // nx)
    below[held] = False
    free = ~below
    free[held] = False
    b = synth.uniform(A.n, 83)
    ref = oracle.solve(A.rowptr, A.colidx, A.vals, b)
    with plan_for(A) as p:
        p.set_spin_limit(1 << 14)
        for algo in ("self", "permuted"):
            p.withhold_row(held)
            got = p.solve(torch.tensor(b, device=dev()), algo=algo).cpu().numpy()
            assert p.status() == (6, held + 1)
            assert relerr(got[free], ref[free]) <= TOL64
            assert np.all(np.isnan(got[below]))
            p.withhold_row(-1)
            assert relerr(p.solve(torch.tensor(b, device=dev()), algo=algo), ref) <= TOL64
            assert p.status() == (0, -1)
