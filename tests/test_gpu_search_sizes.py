"""Batched search at the sizes where a query's share of its cluster changes
(one CTA up to 1024 vertices, then one more per 1024), with bad and pathless
queries beside good ones, against plan_search on the same graphs (cost and path
equal: both follow Dijkstra's tie rule)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # the -m gpu run happens on a GPU machine
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_13507_gb300 import plan as P  # noqa: E402
from paper_2411_13507_gb300 import synth  # noqa: E402


def queries(sizes):
    probs = [synth.triple_integrator_3d(seed=40 + i, N=n, K=max(1, n // 300), nT=3) for i, n in enumerate(sizes)]
    pl = P.Planner.for_problem(probs[0])
    dps = [P.to_device(q, input="f32") for q in probs]
    for dp, q in zip(dps, probs):  # ends at states, so that most queries have a path
        dp.start_pos, dp.goal_pos = q.states[0, :3], q.states[len(q.states) // 2, :3]
    return pl, dps, pl.build_batched(dps)


@pytest.mark.parametrize("sizes", [[1, 2, 37], [1023, 1024, 1025], [2048, 2049, 300, 700], [8192, 8193, 500], [9001, 64]])
def test_equals_single_search(sizes):
    pl, dps, graphs = queries(sizes)
    got = pl.search_batched(dps, graphs)
    single = P.Planner(3, 3, 7, (3.0, 6.0, 30.0), arith="f32", input="f32")
    for r, dp, g in zip(got, dps, graphs):
        one = single.search(dp, g)
        assert r["status"] == one["status"]
        assert r["path"] == one["path"]
        assert r["cost"] == one["cost"] or (np.isinf(r["cost"]) and np.isinf(one["cost"]))


def test_bad_and_short_queries_beside_good_ones():
    pl, dps, graphs = queries([1500, 3000, 400])
    outs = pl.alloc_search_batched(dps)
    bad = P.Graph(N=graphs[0].N, cap=1, **{k: getattr(graphs[0], k) for k in ("row_off", "col", "w", "tidx", "mask", "count")})
    outs[2]["path"] = torch.empty(1, dtype=torch.int32, device="cuda")  # shorter than any path
    pl.prepare_search_batched(dps, [bad, graphs[1], graphs[2]], outs)
    pl.search_batched_async()
    assert pl.wait() == P.PLAN_OK
    ref = pl.search_batched(dps, graphs)
    assert int(outs[0]["status"]) == P.PLAN_ERR_INVALID_ARG
    assert int(outs[1]["status"]) == ref[1]["status"] and float(outs[1]["cost"]) == ref[1]["cost"]
    if ref[2]["path"] and len(ref[2]["path"]) > 1:
        assert int(outs[2]["status"]) == P.PLAN_ERR_CAPACITY and int(outs[2]["path_len"]) == len(ref[2]["path"])


def test_sweep_limit():
    pl, dps, graphs = queries([2500, 900])
    ref = pl.search_batched(dps, graphs)
    pl.set_search_limits(max_sweeps=1)
    outs = pl.alloc_search_batched(dps)
    pl.prepare_search_batched(dps, graphs, outs)
    pl.search_batched_async()
    pl.wait()
    for o, r in zip(outs, ref):
        if r["path"] and len(r["path"]) > 3:
            assert int(o["status"]) == P.PLAN_ERR_TIMEOUT
    pl.set_search_limits()
    again = pl.search_batched(dps, graphs)
    assert [a["path"] for a in again] == [r["path"] for r in ref]
