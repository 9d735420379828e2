"""Batched search on chains 0 -> 1 -> ... -> N-1, whose path, cost and number of
sweeps are known: the statuses OK, CAPACITY and TIMEOUT at the sizes where a
batch changes from one CTA a query to clusters (its largest query above 1024
vertices)."""
import numpy as np
import pytest

from paper_2411_13507_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # the -m gpu run happens on a GPU machine
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_13507_gb300 import plan as P  # noqa: E402


def chain(N, arith):
    prob = synth.double_integrator_2d(seed=1, N=1, K=1, nT=1)
    prob.states = np.zeros((N, 4))
    prob.states[:, 0] = np.arange(N)
    prob.start_pos, prob.goal_pos = np.array([0.0, 0.0]), np.array([N - 1.0, 0.0])
    d = lambda a, t: torch.tensor(a, dtype=t, device="cuda")
    w = 1.0 + (np.arange(N) % 7) / 8.0  # sums of eighths: exact in either type
    g = P.Graph(N=N, cap=N, row_off=d(np.minimum(np.arange(N + 1), N - 1), torch.int32), col=d(np.arange(1, N + 1), torch.int32),
                w=d(w, torch.float64 if arith == "f64" else torch.float32), tidx=d(np.zeros(N), torch.uint8),
                mask=d(np.ones(N), torch.int32), count=d([N - 1], torch.int64))
    return P.to_device(prob, input="f64"), g, float(w[:N - 1].sum())


@pytest.mark.parametrize("arith", ["f64", "f32"])
@pytest.mark.parametrize("sizes", [(2, 31, 1024), (1023,), (1025, 64), (40, 2049), (1, 3)])
def test_statuses(sizes, arith):
    pl = P.Planner(2, 2, 5, (2.0, 4.0), arith=arith, input="f64")
    made = [chain(N, arith) for N in sizes]
    dps, graphs = [x[0] for x in made], [x[1] for x in made]
    for r, N, (_, _, cost) in zip(pl.search_batched(dps, graphs), sizes, made):
        assert r["status"] == P.PLAN_OK and r["path"] == list(range(N)) and r["cost"] == cost
    outs = pl.alloc_search_batched(dps)  # room for all but the last vertex
    for o, N in zip(outs, sizes):
        o["path"] = torch.empty(max(1, N - 1), dtype=torch.int32, device="cuda")
    pl.prepare_search_batched(dps, graphs, outs)
    pl.search_batched_async()
    assert pl.wait() == P.PLAN_OK
    for o, N in zip(outs, sizes):
        assert int(o["status"]) == (P.PLAN_ERR_CAPACITY if N > 1 else P.PLAN_OK) and int(o["path_len"]) == N
    pl.set_search_limits(max_sweeps=2)
    outs = pl.alloc_search_batched(dps)
    pl.prepare_search_batched(dps, graphs, outs)
    pl.search_batched_async()
    pl.wait()
    for o, N in zip(outs, sizes):  # a chain takes N - 1 sweeps that change something, and one that does not
        assert int(o["status"]) == (P.PLAN_ERR_TIMEOUT if N - 1 > 2 else P.PLAN_OK)
    pl.set_search_limits()
    assert [r["status"] for r in pl.search_batched(dps, graphs)] == [P.PLAN_OK] * len(sizes)
