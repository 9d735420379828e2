"""Contexts of several threads, each on its own stream, that call the same
kernels with different amounts of shared memory at the same time: every call
succeeds and gives the single-threaded result."""
import threading

import pytest

from paper_2411_13507_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # the -m gpu run happens on a GPU machine
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_13507_gb300 import plan as P  # noqa: E402


def together(jobs):
    """Runs the jobs in threads of their own, from one start; the exceptions."""
    go, errs = threading.Barrier(len(jobs)), []

    def body(job):
        try:
            go.wait()
            job()
        except Exception as e:  # noqa: BLE001
            errs.append(e)

    ts = [threading.Thread(target=body, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    return errs


def test_closest_points_with_different_rows():
    points = torch.rand((40, 2), device="cuda") * 20.0
    jobs, checks = [], []
    for n, cuts in ((32, 0), (128, 3)):
        pl = P.Planner(2, 2, 5, (2.0, 4.0), arith="f32", input="f32", stream=torch.cuda.Stream())
        obst = P.obstacles_to_device(synth.obstacles(2, n, 2, max_cuts=cuts), input="f32")
        torch.cuda.synchronize()
        pl.wait()
        want = pl.obstacle_planes(points, obst)
        out = {k: torch.empty_like(v) for k, v in want.items()}

        def job(pl=pl, obst=obst, out=out):
            for _ in range(4000):
                pl.obstacle_planes_async(points, obst, out)

        jobs.append(job)
        checks.append((pl, want, out))
    torch.cuda.synchronize()
    assert together(jobs) == []
    for pl, want, out in checks:
        assert pl.wait() == P.PLAN_OK
        assert all(torch.equal(want[k], out[k]) for k in want)


def test_builds_with_different_tiles_and_costs():
    jobs, checks = [], []
    for n, tile, cost in ((60, 8, "pos"), (2000, 64, "state")):
        prob = synth.triple_integrator_3d(seed=3, N=n, K=8, nT=2)
        prob.model.cost_mode = cost
        pl = P.Planner.for_problem(prob, arith="f32", input="f32", stream=torch.cuda.Stream())
        pl.set_tile(tile=tile)
        dp = P.to_device(prob, input="f32")
        torch.cuda.synchronize()
        want = pl.build_edges(dp)
        out = pl.alloc_graph(want.N, max(1, want.E))

        def job(pl=pl, dp=dp, out=out):
            for _ in range(400):
                pl.build_edges_async(dp, out)

        jobs.append(job)
        checks.append((pl, want.to_numpy(), out))
    torch.cuda.synchronize()
    assert together(jobs) == []
    for pl, want, out in checks:
        assert pl.wait() == P.PLAN_OK
        got = out.to_numpy()
        assert all((want[k] == got[k]).all() for k in want)
