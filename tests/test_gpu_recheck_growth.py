"""A first build whose re-check list overflows far above its first size (65,536
entries) grows it within the retries of build_edges: the precision forms on many
states that share every polytope, whose masks must equal the FP64 form's."""
import numpy as np
import pytest

from paper_2411_13507_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # the -m gpu run happens on a GPU machine
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_13507_gb300 import plan as P  # noqa: E402


@pytest.mark.parametrize("arith,m", [("tf32", 2), ("bf16", 2)])
def test_many_open_margins(arith, m):
    prob = synth.double_integrator_2d(seed=3, N=1200, K=4, nT=16)
    prob.states[:, :2] = 5.0 + np.random.default_rng(3).uniform(-0.5, 0.5, (1200, 2))
    prob.A = np.tile(np.concatenate([np.eye(2), -np.eye(2)]), (4, 1))
    prob.b = np.concatenate([[5.0 + h, 5.0 + h, h - 5.0, h - 5.0] for h in (0.55, 0.6, 0.7, 0.8)])
    prob.poly_off = (4 * np.arange(5)).astype(np.int32)
    dp = P.to_device(prob, input="f64")
    want = P.Planner.for_problem(prob, arith="f64", input="f64").build_edges(dp).to_numpy()
    pl = P.Planner.for_problem(prob, arith=arith, input="f64")
    got = pl.build_edges(dp).to_numpy()
    assert pl.info()["rechecks"] > 10 * 65536
    assert all(np.array_equal(got[k], want[k]) for k in ("row_off", "col", "mask"))
