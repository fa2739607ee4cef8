"""A value that never comes, where the rows that do not need it are the most
exposed: a launch of so few warps that they own every ticket."""
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
