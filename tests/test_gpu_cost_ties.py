"""FP64 weights where the FP32 costs cannot tell the durations apart: repeated
durations (exact ties go to the lower index), durations a few units in the last
place or 1e-7 apart, and states that nearly coincide.  The default FP64 route
must equal the canonical FP64 pair kernel (pipeline 3) bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # the -m gpu run happens on a GPU machine
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_13507_gb300 import plan as P  # noqa: E402
from paper_2411_13507_gb300 import synth  # noqa: E402


@pytest.mark.parametrize("m,p", [(2, 3), (2, 5), (3, 5), (3, 7)])
@pytest.mark.parametrize("kind", ["repeated", "ulp", "close", "one", "coincident"])
@pytest.mark.parametrize("cost", ["state", "pos"])
def test_equal_to_the_canonical_route(m, p, kind, cost):
    f = synth.double_integrator_2d if m == 2 else synth.triple_integrator_3d
    prob = f(seed=3, N=90, K=2, nT=4, degree=p, dtype="f64")
    prob.model.cost_mode = cost
    base = np.array([0.8, 1.3, 2.1])
    prob.T = {"repeated": np.repeat(base, 3), "ulp": np.concatenate([base, np.nextafter(base, 9), base * (1 + 2e-15)]),
              "close": np.concatenate([base * (1 + 1e-7), base]), "one": base[:1], "coincident": base}[kind]
    if kind == "coincident":
        prob.states[1::2] = prob.states[0::2] * (1 + 1e-9)
    dp = P.to_device(prob, input="f64")
    got = []
    for pipeline in (0, 3):
        pl = P.Planner.for_problem(prob, arith="f64", input="f64")
        pl.set_tile(pipeline=pipeline)
        got.append(pl.build_edges(dp).to_numpy())
    assert all(np.array_equal(got[0][k], got[1][k]) for k in got[0])
