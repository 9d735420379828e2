"""Membership and compaction where their groups of 32 end: member counts and
state counts around 32 and 128, words of 32 polytopes, states in more than 32
polytopes, rows with more entries than the staged path holds, empty queries in
a batch.  Graphs equal the FP64 oracle's."""
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


def check(prob, arith="f32"):
    pl = P.Planner.for_problem(prob, arith=arith)
    g = pl.build_edges(P.to_device(prob, input=prob.dtype))
    csr = oracle.OracleProblem(prob).csr(with_detail=True)
    parity.compare_full(g.to_numpy(), csr, prob.N, prob.nT, arith)
    assert pl.info()["candidates"] == csr["candidates"]
    return g


def boxes(prob, centres, half):
    """The problem's polytopes replaced by axis boxes."""
    m = prob.model.m
    A = np.concatenate([np.eye(m), -np.eye(m)])
    prob.A = np.tile(A, (len(centres), 1))
    prob.b = np.concatenate([np.concatenate([c + half, half - c]) for c in centres])
    prob.poly_off = (2 * m * np.arange(len(centres) + 1)).astype(np.int32)
    return prob


@pytest.mark.parametrize("N", [1, 31, 32, 33, 64, 127, 128, 129, 257])
def test_member_counts(N):
    check(synth.double_integrator_2d(2, N=N, K=1, nT=3), "f64")


@pytest.mark.parametrize("K", [31, 32, 33, 64, 65, 97])
def test_words_of_polytopes(K):
    check(synth.double_integrator_2d(4, N=150, K=K, nT=2), "f64")


@pytest.mark.parametrize("K,same", [(3, True), (33, True), (40, True), (40, False), (70, False)])
def test_states_in_many_polytopes(K, same):
    prob = synth.double_integrator_2d(5, N=90, K=1, nT=2)
    rng = np.random.default_rng(K)
    c = prob.states[:, :2].mean(0)
    boxes(prob, [c if same else c + rng.uniform(-1.0, 1.0, 2) for _ in range(K)], 2.0)
    check(prob, "f64")


def test_long_shared_rows():
    """Every state in two polytopes and rows of over 512 entries."""
    prob = synth.double_integrator_2d(6, N=700, K=1, nT=1)
    prob.T = np.array([1.9])
    rng = np.random.default_rng(6)
    prob.states[:, :2] = rng.uniform(4.0, 6.0, (700, 2))
    prob.states[:, 2:] *= 0.2
    boxes(prob, [np.array([5.0, 5.0]), np.array([5.1, 4.9])], 1.5)
    g = check(prob, "f64")
    assert int(torch.diff(g.row_off).max()) > 512


def test_batch_of_uneven_and_empty_queries():
    probs = [synth.triple_integrator_3d(seed=70 + i, N=n, K=k, nT=3) for i, (n, k) in
             enumerate([(1, 1), (33, 2), (0, 3), (300, 40), (5, 0), (64, 64), (129, 1)])]
    pl = P.Planner.for_problem(probs[0])
    graphs = pl.build_batched([P.to_device(q, input="f32") for q in probs])
    for q, g in zip(probs, graphs):
        if q.N == 0 or q.K == 0:
            assert g.E == 0
            continue
        parity.compare_full(g.to_numpy(), oracle.OracleProblem(q).csr(with_detail=True), q.N, q.nT, "f32")
