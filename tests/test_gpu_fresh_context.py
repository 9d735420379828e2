"""A context's first call sees a clean status word, whatever the memory held
before: closest points as the first call of new contexts, made where contexts
that ended with an error status have been released."""
import pytest

from paper_2411_13507_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # the -m gpu run happens on a GPU machine
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_13507_gb300 import plan as P  # noqa: E402


def test_first_call_after_a_failed_context():
    prob = synth.double_integrator_2d(seed=1, N=64, K=1, nT=1)
    prob.T = prob.T[:1] * 1e-3  # too short for any edge: no path
    dp = P.to_device(prob, input="f64")
    points = torch.rand((50, 2), device="cuda") * 20.0
    obst = P.obstacles_to_device(synth.obstacles(1, 40, 2), input="f32")
    for _ in range(6):
        bad = P.Planner.for_problem(prob, arith="f64", input="f64")
        g = bad.build_edges(dp)
        assert g.E == 0
        bad.search_async(dp, g, prob.states[0, :2], prob.states[1, :2], bad.alloc_search(prob.N))
        torch.cuda.synchronize()
        bad.close()  # its status word says NO_PATH
        new = P.Planner(2, 2, 5, (2.0, 4.0), arith="f32", input="f32")
        new.obstacle_planes(points, obst)
        new.close()
