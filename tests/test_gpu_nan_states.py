"""States with NaN among their derivatives: the FP32 pair kernels (screened, warp-specialised,
every pair through all rows) give the same graph, whatever polytope rows lie
along an axis."""
import numpy as np
import pytest

from paper_2411_13507_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # the -m gpu run happens on a GPU machine
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_13507_gb300 import plan as P  # noqa: E402


@pytest.mark.parametrize("m,p", [(2, 3), (2, 5), (3, 5), (3, 7)])
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("order", [1, "last"])
@pytest.mark.parametrize("seed", [1, 2, 3])
def test_kernels_agree(m, p, axis, order, seed):
    f = synth.double_integrator_2d if m == 2 else synth.triple_integrator_3d
    prob = f(seed=seed, N=180, K=2, nT=4, degree=p, dtype="f32")
    prob.T = np.array([0.5, 1.0, 1.5, 2.5])
    prob.states[::4, (m - 1 if order == "last" else order) * m + axis] = np.nan
    dp = P.to_device(prob, input="f32")
    got = []
    for pipeline in (0, 1, 2):
        pl = P.Planner.for_problem(prob, arith="f32", input="f32")
        pl.set_tile(pipeline=pipeline)
        got.append(pl.build_edges(dp).to_numpy())
    nan = np.isnan(prob.states).any(1)
    rows = np.repeat(np.arange(prob.N), np.diff(got[2]["row_off"]))
    assert np.any(nan[rows] | nan[got[2]["col"]])  # some edges of theirs are decided by the other axes
    for g in got[:2]:
        assert all(np.array_equal(g[k], got[2][k]) for k in ("row_off", "col", "mask"))
