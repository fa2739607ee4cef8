"""Calls that a rule sends to the wrong kernel cost many times what the right one
takes.  Each is held against a call on the same system that takes the other way: the
bounds leave a factor of two or more between what is measured and what fails."""
import numpy as np
import pytest
import torch

import synth
from gpu_util import dev, plan_for

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu(cuda_device):
    yield


def _dense(n):
    i, j = np.tril_indices(n)
    return synth._from_sorted_coo(n, i, j, np.where(i == j, 2.0 * n, -1.0), upper=False)


def _band(n, width):
    i = np.repeat(np.arange(n), width + 1)
    j = i - np.tile(np.arange(width, -1, -1), n)
    i, j = i[j >= 0], j[j >= 0]
    return synth._from_sorted_coo(n, i, j, np.where(i == j, 2.0 * width, -1.0), upper=False)


def _ms(call, reps=5):
    times = []
    for _ in range(reps + 1):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    return min(times[1:])


@pytest.mark.parametrize("algo", ["self", "permuted"])
@pytest.mark.parametrize("make", [lambda: _dense(1500), lambda: _band(8000, 70)])
def test_tickets_of_long_rows_that_straddle_levels(make, algo):
    """One row a level, several chunks a row: with 8 and 16 lanes about as fast as with
    32, where a ticket is one row, and 16 columns about as fast as 8."""
    A = make()
    b = torch.tensor(synth.uniform((A.n, 16), 3), device=dev())
    one, few = b[:, 0].contiguous(), b[:, :8].contiguous()
    with plan_for(A) as p:
        p.set_tuning(32, 256, 304)
        whole = _ms(lambda: p.solve(one, algo=algo))
        for lanes in (8, 16):
            p.set_tuning(lanes, 256, 304)
            assert _ms(lambda: p.solve(one, algo=algo)) < 3.0 * whole, lanes
            assert _ms(lambda: p.solve_transpose(one)) < 3.0 * whole, lanes
        assert _ms(lambda: p.solve(b, algo=algo)) < 3.0 * _ms(lambda: p.solve(few, algo=algo))


@pytest.mark.parametrize("lanes", [1, 2])
def test_partitioned_solve_of_rows_that_differ(lanes):
    """Parts of twenty rows, a row a group, up to a thousand entries of earlier parts: the
    sliced copy would take two to three times as long as the level-ordered one."""
    A = synth.general_lower(3001, 5)
    b = torch.tensor(synth.uniform(A.n, 3), device=dev())
    with plan_for(A) as p:
        p.set_tuning(lanes, 256, 0)
        assert torch.equal(p.solve(b, algo="partitioned"), p.solve(b, algo="self"))
        assert (_ms(lambda: p.solve(b, algo="partitioned"))
                < 1.5 * _ms(lambda: p.solve(b, algo="permuted")))


def test_partitioned_solve_with_a_warp_per_short_row():
    """32 lanes on rows of two entries: in place, not on the level-ordered copy, which
    would take nearly twice as long."""
    A = synth.lap2d_5pt_lower(1024, 1024)
    b = torch.tensor(synth.uniform(A.n, 3), device=dev(), dtype=torch.float32)
    with plan_for(A, dtype=torch.float32) as p:
        p.set_tuning(32, 512, 0)
        p.set_partition(4096, 4)
        want = p.solve(b, algo="self")
        assert torch.equal(p.solve(b, algo="partitioned"), want)
        x = b.clone()
        assert torch.equal(p.solve(x, out=x, algo="partitioned"), want)
        assert (_ms(lambda: p.solve(b, algo="partitioned"))
                < 1.4 * _ms(lambda: p.solve(b, algo="self")))
        p.prepare("partitioned")
        x = b.clone()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            p.solve(x, out=x, algo="partitioned")
        g.replay()
        assert torch.equal(x, want)


def test_partitioned_solve_of_wide_levels_and_empty_slots():
    A = synth.lap3d_7pt_lower(96, 96, 96)
    b = torch.tensor(synth.uniform(A.n, 3), device=dev())
    with plan_for(A) as p:
        p.set_tuning(16, 512, 0)
        p.set_partition(4096, 4)
        assert torch.equal(p.solve(b, algo="partitioned"), p.solve(b, algo="self"))
        assert (_ms(lambda: p.solve(b, algo="partitioned"))
                < 1.4 * _ms(lambda: p.solve(b, algo="permuted")))


def test_partitioned_solve_of_many_general_systems():
    """Wide levels because the systems are many: the slices take a third less than the
    level-ordered copy (systems of all sizes: two thirds less)."""
    A = synth.block_diagonal([synth.general_lower(4000, 5)] * 200)
    b = torch.tensor(synth.uniform(A.n, 3), device=dev())
    with plan_for(A) as p:
        p.set_tuning(8, 512, 0)
        assert torch.equal(p.solve(b, algo="partitioned"), p.solve(b, algo="self"))
        assert (_ms(lambda: p.solve(b, algo="partitioned"))
                < 0.8 * _ms(lambda: p.solve(b, algo="permuted")))
