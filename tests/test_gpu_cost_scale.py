"""FP64 weights at the ends of the FP32 range: a problem scaled by a power of two
(states, polytopes and bounds) scales every FP64 product, sum and root exactly,
so its graph must have the unscaled problem's masks and durations and its weights
times the scale, and the default FP64 route must equal the canonical FP64 pair
kernel (pipeline 3) bit for bit -- also where FP32 squares of the rows underflow
(below 2^-75) or overflow (above 2^64)."""
import numpy as np
import pytest

from paper_2411_13507_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # the -m gpu run happens on a GPU machine
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_13507_gb300 import plan as P  # noqa: E402


def graph(prob, pipeline):
    pl = P.Planner.for_problem(prob, arith="f64", input="f64")
    pl.set_tile(pipeline=pipeline)
    return pl.build_edges(P.to_device(prob, input="f64")).to_numpy()


@pytest.mark.parametrize("m,p", [(2, 5), (3, 7)])
@pytest.mark.parametrize("cost", ["state", "pos"])
@pytest.mark.parametrize("k", [-80, -72, -66, -62, -58, -40, 58, 60, 61, 62, 63, 64, 68])
def test_scaled_problem(m, p, cost, k):
    f = synth.double_integrator_2d if m == 2 else synth.triple_integrator_3d
    prob = f(seed=9, N=250, K=2, nT=4, degree=p, dtype="f64")
    prob.model.cost_mode = cost
    prob.T = np.array([0.8, 1.3, 2.1, 2.9])
    one = graph(prob, 3)
    assert np.any(one["mask"] & (one["mask"] - 1))  # edges with several durations
    s = 2.0 ** k
    prob.states, prob.b = prob.states * s, prob.b * s
    prob.model.bounds = tuple(c * s for c in prob.model.bounds)
    want, got = graph(prob, 3), graph(prob, 0)
    assert all(np.array_equal(want[x], got[x]) for x in want)
    assert all(np.array_equal(one[x], got[x]) for x in ("row_off", "col", "mask", "t"))
    assert np.array_equal(one["w"] * s, got["w"])
