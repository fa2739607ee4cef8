"""The multi-RHS kernel's ways of taking a ticket's rows: rows of at most one
chunk of entries, longer ones, and rows of very different lengths; tickets that
straddle levels; more and fewer columns than lanes; a row that is withheld.
Every column is folded in one fixed order, so a result must not depend on the
width, the grid or the form."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import TOL32, TOL64, bidiagonal, dev, diagonal, long_rows, plan_for, relerr, \
    unit_without_diagonal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu(cuda_device):
    yield


MATRICES = {
    "short_ilu_unit": lambda: synth.lap3d_7pt_ilu0(9, 7, 8)[0],      # one chunk, unit diagonal
    "short_ilu_upper": lambda: synth.lap3d_7pt_ilu0(9, 7, 8)[1],
    "nine_point": lambda: synth.laplacian_triangles((23, 19), 9)[0],  # a chunk and the diagonal
    "grid27": lambda: synth.laplacian_triangles((7, 6, 9), 27)[1],   # four chunks
    "chain": lambda: bidiagonal(300),
    "diagonal": lambda: diagonal(70),
    "apart": lambda: long_rows(3000),
    "unit_nodiag": lambda: unit_without_diagonal(),
}


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("k", [2, 5, 17, 33])
@pytest.mark.parametrize("name", sorted(MATRICES))
def test_columns_do_not_depend_on_the_shape(name, k, dtype):
    A = MATRICES[name]()
    b = synth.uniform((A.n, k), 91)
    tol = TOL64 if dtype == torch.float64 else TOL32
    bt = torch.tensor(b, device=dev(), dtype=dtype)
    with plan_for(A, dtype=dtype) as p:
        first = p.solve(bt)
        first_t = p.solve_transpose(bt)
        for j in (0, k // 2, k - 1):
            ref = oracle.solve(A.rowptr, A.colidx, A.vals, b[:, j].copy(), upper=A.upper,
                               unit=A.unit)
            assert relerr(first[:, j].double(), ref) <= tol, j
        for lanes in (4, 8, 16, 32):
            for block, cap in ((64, 1), (256, 0), (1024, 2)):
                p.set_mrhs_tuning(lanes, block, cap)
                assert torch.equal(p.solve(bt), first), (lanes, block)
                assert torch.equal(p.solve(bt, algo="permuted"), first), (lanes, block)
            assert torch.equal(p.solve_transpose(bt), first_t), lanes
            x = bt.clone()
            assert torch.equal(p.solve(x, out=x), first)
        wide = torch.zeros(A.n, k + 3, device=dev(), dtype=dtype)   # a leading dimension
        wide[:, :k] = bt
        out = torch.full_like(wide, 7.0)
        p.solve(wide[:, :k], out=out[:, :k])
        assert torch.equal(out[:, :k], first) and torch.all(out[:, k:] == 7.0)
        assert p.status() == (0, -1)


@pytest.mark.parametrize("algo", ["self", "permuted"])
@pytest.mark.parametrize("make", ["alike", "apart"])
def test_a_withheld_row_holds_up_only_its_dependents(algo, make):
    if make == "alike":
        A = synth.lap2d_5pt_lower(30, 60)
    else:
        A = synth.block_diagonal([synth.general_lower(900, 5), synth.general_lower(2500, 6)])
    held = 500
    reach = np.zeros(A.n, dtype=bool)
    reach[held] = True
    for i in range(held + 1, A.n):
        reach[i] = reach[A.colidx[A.rowptr[i]:A.rowptr[i + 1] - 1]].any()
    free = ~reach
    reach[held] = False
    b = synth.uniform((A.n, 5), 93)
    ref = np.stack([oracle.solve(A.rowptr, A.colidx, A.vals, b[:, j].copy()) for j in range(5)], 1)
    with plan_for(A) as p:
        p.set_spin_limit(1 << 14)
        p.withhold_row(held)
        got = p.solve(torch.tensor(b, device=dev()), algo=algo).cpu().numpy()
        assert p.status() == (6, int(np.flatnonzero(reach)[0]))
        assert relerr(got[free], ref[free]) <= TOL64
        assert np.all(np.isnan(got[reach]))
        p.withhold_row(-1)
        assert relerr(p.solve(torch.tensor(b, device=dev()), algo=algo), ref) <= TOL64
        assert p.status() == (0, -1)
