"""A value that never comes, where the rows that do not need it are the most
exposed: a launch of so few warps that they own every ticket, and a chain that goes
on for many windows of the one-cluster kernel after the missing row."""
import time

import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import TOL64, dev, plan_for, relerr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu(cuda_device):
    yield


def _behind(A, held):
    """Rows that need row `held`."""
    reach = np.zeros(A.n, dtype=bool)
    reach[held] = True
    for i in range(held + 1, A.n):
        reach[i] = reach[A.colidx[A.rowptr[i]:A.rowptr[i + 1] - 1]].any()
    reach[held] = False
    return reach


@pytest.mark.parametrize("lanes", [4, 32])
@pytest.mark.parametrize("algo", ["self", "permuted"])
@pytest.mark.parametrize("make", ["alike", "apart"])
def test_two_warps_that_own_every_ticket(make, algo, lanes):
    if make == "alike":
        A = synth.lap2d_5pt_lower(30, 60)
    else:
        A = synth.block_diagonal([synth.general_lower(900, 5), synth.general_lower(2500, 6)])
    held = 500
    behind = _behind(A, held)
    free = ~behind
    free[held] = False
    b = synth.uniform((A.n, 5), 93)
    ref = np.stack([oracle.solve(A.rowptr, A.colidx, A.vals, b[:, j].copy()) for j in range(5)], 1)
    with plan_for(A) as p:
        p.set_mrhs_tuning(lanes, 64, 1)
        p.set_spin_limit(1 << 12)
        p.withhold_row(held)
        got = p.solve(torch.tensor(b, device=dev()), algo=algo).cpu().numpy()
        assert p.status() == (6, int(np.flatnonzero(behind)[0]))
        assert np.all(np.isnan(got[behind]))
        assert relerr(got[free], ref[free]) <= TOL64


def _braid(n, held):
    """Rows 3 i and 3 i + 1 are two chains, row 3 i + 2 a leaf of the first one; of
    the leaves past `held` (in the second chain) every 50th needs row `held` too."""
    i = np.arange(n)
    first, second = i[3:][i[3:] % 3 == 0], i[3:][i[3:] % 3 == 1]
    leaf = i[i % 3 == 2]
    far = leaf[(leaf > held) & (leaf // 3 % 50 == 0)]
    r = np.concatenate([i, first, second, leaf, far])
    c = np.concatenate([i, first - 3, second - 3, leaf - 2, np.full(far.size, held)])
    order = np.lexsort((c, r))
    r, c = r[order], c[order]
    return synth._from_sorted_coo(n, r, c, np.where(r == c, 2.0, -1.0), upper=False), far


@pytest.mark.parametrize("algo", ["self", "permuted"])
@pytest.mark.parametrize("lanes", [16, 32])
def test_windows_after_a_missing_value_run_as_usual(lanes, algo):
    """The rows of 40 windows that do not need the missing value are exact, and the
    call takes a few times what one takes in which nothing is missing (0.1 s; seconds
    if every level goes through its whole window)."""
    held = 4999                                        # in the first window
    A, far = _braid(40 * 12288 + 100, held)
    behind = np.zeros(A.n, dtype=bool)
    behind[held + 3::3] = True                         # the second chain, and
    behind[far] = True
    free = ~behind
    free[held] = False
    b = synth.uniform(A.n, 97)
    ref = oracle.solve(A.rowptr, A.colidx, A.vals, b)
    bt = torch.tensor(b, device=dev())
    with plan_for(A) as p:
        p.set_tuning(lanes, 256, 0)
        p.set_spin_limit(1 << 12)
        assert relerr(p.solve(bt, algo=algo), ref) <= TOL64   # the copy is built
        assert p.last_launch_count == 1                # one cluster (too large for one block)
        p.withhold_row(held)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        got = p.solve(bt, algo=algo).cpu().numpy()
        assert time.perf_counter() - t0 < 1.0
        assert p.status() == (6, int(np.flatnonzero(behind)[0]))
        assert np.all(np.isnan(got[behind]))
        assert relerr(got[free], ref[free]) <= TOL64
        p.withhold_row(-1)
        assert relerr(p.solve(bt, algo=algo), ref) <= TOL64
        assert p.status() == (0, -1)
