"""The sliced copies of several widths: what is kept, what an update of the values costs,
and that every solve, also a captured one, sees the new values."""
import pytest
import torch

import oracle
import synth
from gpu_util import TOL64, dev, long_rows, plan_for, relerr, unit_without_diagonal

pytestmark = pytest.mark.gpu
WIDTHS = (1, 2, 4, 8, 16)


@pytest.fixture(scope="module", autouse=True)
def _gpu(cuda_device):
    yield


def _ms(call, reps=7):
    times = []
    for _ in range(reps + 1):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    return min(times[1:])


MATRICES = {
    "ilu_upper": lambda: synth.lap3d_7pt_ilu0(21, 23, 19)[1],
    "grid27": lambda: synth.laplacian_triangles((13, 12, 17), 27)[0],
    "long_rows": lambda: long_rows(),
    "unit_nodiag": lambda: unit_without_diagonal(),
}


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("name", sorted(MATRICES))
def test_new_values_after_solves_at_several_widths(name, dtype):
    A = MATRICES[name]()
    b = torch.tensor(synth.uniform(A.n, 61), device=dev(), dtype=dtype)
    with plan_for(A, dtype=dtype) as p:
        p.set_partition(4096, 1)
        graphs = {}
        for lanes in WIDTHS:
            p.set_tuning(lanes, 256, 0)
            p.solve(b, algo="partitioned")
            p.solve_transpose(b, algo="partitioned")
            if lanes in (2, 8):              # of these two, one was not prepared
                if lanes == 2:
                    p.prepare("partitioned")
                x = torch.empty_like(b)
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g):
                    p.solve(b, out=x, algo="partitioned")
                graphs[lanes] = (g, x)
        for factor in (2.0, 0.5):
            p.set_values(factor * p.vals)
            for lanes, (g, x) in graphs.items():
                p.set_tuning(lanes, 256, 0)
                g.replay()
                assert torch.equal(x, p.solve(b, algo="self")), lanes
            for lanes in WIDTHS:
                p.set_tuning(lanes, 256, 0)
                assert torch.equal(p.solve(b, algo="partitioned"), p.solve(b, algo="self")), lanes
                assert torch.equal(p.solve_transpose(b, algo="partitioned"),
                                   p.solve_transpose(b, algo="self")), lanes
        if dtype == torch.float64:
            p.best_algo = "partitioned"
            ref = oracle.solve(A.rowptr, A.colidx, A.vals, b.cpu().numpy(), upper=A.upper,
                               unit=A.unit)
            for lanes in (4, 1, 4):
                p.set_tuning(lanes, 256, 0)
                p.set_values(p.vals.clone())
                assert relerr(p.solve_refined(b)[0], ref) <= TOL64
        assert p.status() == (0, -1)


def test_an_update_pays_for_the_width_in_use():
    A = synth.lap3d_7pt_ilu0(96, 96, 96)[0]
    b = torch.tensor(synth.uniform(A.n, 63), device=dev())
    with plan_for(A) as p, plan_for(A) as q:
        for plan, widths in ((p, (4,)), (q, (1, 2, 8, 4))):
            for lanes in widths:
                plan.set_tuning(lanes, 256, 0)
                plan.solve(b, algo="partitioned")
        one = _ms(lambda: p.set_values(p.vals))
        several = _ms(lambda: q.set_values(q.vals))
        assert several < 1.5 * one


def test_copies_of_several_widths_are_bounded():
    """Together at most as many slots as one copy may have (8 per entry and 2^20), each
    with a value and a column; here the widths would take 12 slots per entry."""
    A = synth.lap2d_5pt_lower(1500, 1500)
    b = torch.tensor(synth.uniform(A.n, 65), device=dev())
    with plan_for(A) as p:
        p.set_partition(8192, 1)
        p.set_tuning(1, 256, 0)
        want = p.solve(b, algo="partitioned")
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        for lanes in (2, 4, 8, 16):
            p.set_tuning(lanes, 256, 0)
            p.solve(b, algo="partitioned")
        torch.cuda.synchronize()
        # beside the slots 1/d and the descriptors of the groups (at least two rows each,
        # six at few lanes)
        beside = 4 * 8 * A.n + 16 * (A.n // 2 + A.n // 3 + 2 * A.n // 6)
        assert free - torch.cuda.mem_get_info()[0] <= 12 * (8 * A.nnz + 2**20) + beside
        p.set_tuning(1, 256, 0)
        assert torch.equal(p.solve(b, algo="partitioned"), want)


def test_an_update_of_long_rows():
    """About as long as that of the level-ordered copy (three times as long, one entry
    after the other)."""
    A = synth.general_lower(3001, 5)
    b = torch.tensor(synth.uniform(A.n, 67), device=dev())
    with plan_for(A) as p, plan_for(A) as q:
        p.set_tuning(16, 256, 0)
        p.set_partition(4096, 1)
        p.solve(b, algo="partitioned")
        q.solve(b, algo="permuted")
        assert _ms(lambda: p.set_values(p.vals)) < 2.0 * _ms(lambda: q.set_values(q.vals))


def test_a_recorded_update_covers_every_copy_on_every_replay():
    """New values and a solve at one width in a graph; solves at another width, and on the
    level-ordered copy, see the values of each replay, also once their copies had to make
    room for others'."""
    A = synth.lap3d_7pt_ilu0(21, 23, 19)[0]
    b = torch.tensor(synth.uniform(A.n, 69), device=dev())
    with plan_for(A) as p:
        for lanes in (2, 4):
            p.set_tuning(lanes, 256, 0)
            p.solve(b, algo="partitioned")
        p.solve(b, algo="permuted")
        x = torch.empty_like(b)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            p.vals.mul_(2.0)
            p.refresh_values()
            p.solve(b, out=x, algo="partitioned")
        for lanes in (1, 8, 16):             # other copies, after the capture
            p.set_tuning(lanes, 256, 0)
            p.solve(b, algo="partitioned")
        for _ in range(3):
            g.replay()
            for lanes in (2, 4):
                p.set_tuning(lanes, 256, 0)
                want = p.solve(b, algo="self")
                assert torch.equal(p.solve(b, algo="partitioned"), want), lanes
                assert torch.equal(p.solve(b, algo="permuted"), want), lanes
            assert torch.equal(x, want)


def test_captured_solves_of_a_prepared_width_follow_to_another_array_of_values():
    """At 32 lanes on rows of two entries (in place unless captured) as at two."""
    A = synth.lap2d_5pt_lower(400, 410)
    b = torch.tensor(synth.uniform(A.n, 71), device=dev())
    with plan_for(A) as p:
        p.set_partition(4096, 1)
        graphs = []
        for lanes in (2, 32):
            p.set_tuning(lanes, 256, 0)
            p.prepare("partitioned")
            x = b.clone()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                p.solve(x, out=x, algo="partitioned")
            graphs.append((lanes, g, x))
        first = p.vals
        p.set_values(2.0 * first)
        first.fill_(float("nan"))             # nobody reads it any more
        for lanes, g, x in graphs:
            p.set_tuning(lanes, 256, 0)
            x.copy_(b)
            g.replay()
            assert torch.equal(x, p.solve(b, algo="self")), lanes
            assert torch.equal(x, p.solve(b, algo="partitioned")), lanes
