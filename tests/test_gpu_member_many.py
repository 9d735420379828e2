"""Membership of many states by staged rows (k_member_many, taken from four
groups of 256 states and a word of 32 polytopes a multiprocessor) against the
form that single queries take: batches of small uneven queries around both group
sizes, with empty ones among them, whose graphs must equal the single builds'
bit for bit, and the FP64 oracle's."""
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

SIZES, COUNTS = (0, 1, 255, 256, 257), (0, 1, 32, 33, 130)


def query(m, N, K, seed):
    f = synth.double_integrator_2d if m == 2 else synth.triple_integrator_3d
    q = f(seed=seed, N=max(N, 1), K=max(K, 1), nT=2, dtype="f64" if m == 2 else "f32")
    q.states = q.states[:N]
    if K == 0:
        q.poly_off, q.A, q.b = q.poly_off[:1], q.A[:0], q.b[:0]
    return q


@pytest.mark.parametrize("m,arith", [(2, "f64"), (2, "f32"), (3, "f32"), (3, "f64")])
def test_batch_equals_single_builds(m, arith):
    sizes = [(N, K) for N in SIZES for K in COUNTS] * 4
    probs = [query(m, N, K, 100 + i) for i, (N, K) in enumerate(sizes)]
    mask = sum(N * max(1, (K + 31) // 32) for N, K in sizes)
    groups = mask // 256 + len(sizes) * ((max(COUNTS) + 31) // 32 + 2)
    assert groups >= 4 * torch.cuda.get_device_properties(0).multi_processor_count  # the batch takes the form in question
    store = "f64" if m == 2 else "f32"
    pl = P.Planner.for_problem(probs[0], arith=arith, input=store)
    single = P.Planner.for_problem(probs[0], arith=arith, input=store)
    dps = [P.to_device(q, input=store) for q in probs]
    graphs = pl.build_batched(dps)
    edges = 0
    for i, (q, dp, g) in enumerate(zip(probs, dps, graphs)):
        got, one = g.to_numpy(), single.build_edges(dp).to_numpy()
        assert all(np.array_equal(got[k], one[k]) for k in one)
        if i < len(SIZES) * len(COUNTS) and q.N and q.K:
            parity.compare_full(got, oracle.OracleProblem(q).csr(with_detail=True), q.N, q.nT, arith)
        edges += g.E
    assert edges > 1000
