"""Both sides of the screened pair kernel's choices in one tile: durations with
enough feasible pairs for staged costs (160) beside durations with a few, and
durations whose rows leave the FP16 range beside ordinary ones; which of them
occur is asserted from the oracle's graph and the tables.  Graphs equal the FP64
oracle's (masks and edges exactly, weights within 1e-5)."""
import numpy as np
import pytest

import oracle
import parity
from paper_2411_13507_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # the -m gpu run happens on a GPU machine
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_13507_gb300 import plan as P  # noqa: E402

SC_STAGE, FP16_ROWS = 160, 2.0 ** 14


@pytest.mark.parametrize("m,p", [(2, 3), (2, 5), (3, 5), (3, 7)])
@pytest.mark.parametrize("cost", ["state", "pos"])
def test_staged_and_scaled(m, p, cost):
    f = synth.double_integrator_2d if m == 2 else synth.triple_integrator_3d
    prob = f(4, N=64, K=1, degree=p, nT=4)
    prob.T = np.concatenate([[0.002, 0.01], np.linspace(0.4, 4.0, 19)]).astype(np.float32).astype(np.float64)
    prob.model.cost_mode = cost
    csr = oracle.OracleProblem(prob).csr(with_detail=True)
    n = np.array([np.count_nonzero((csr["mask"] >> t) & 1) for t in range(prob.nT)])
    assert np.any(n >= SC_STAGE) and np.any((n > 0) & (n < SC_STAGE)), n
    H = P.model_tables(m, p, prob.T)["H"]
    rows = [p - k + 1 for k in range(1, m + 1)]
    lim = np.repeat(prob.model.bounds, rows)
    size = np.abs(H / lim[None, :, None]).max(axis=(1, 2)) * np.abs(prob.states[:, :m] - prob.states[0, :m]).max()
    assert size[0] > FP16_ROWS and size[-1] < FP16_ROWS, size
    pl = P.Planner.for_problem(prob, arith="f32")
    g = pl.build_edges(P.to_device(prob, input=prob.dtype)).to_numpy()
    parity.compare_full(g, csr, prob.N, prob.nT, "f32")
