"""Refinement loss and gradients for bounds and relaxation points so small that
products of two margins, or the square of the relaxation point, leave the FP32
range.  Against the FP64 oracle, within 1e-3 of the output's largest value: the
slopes 1 / (c - Q) - 1 / (c + Q) lose up to c / |Q| (about 10 here) of their
FP32 digits, and up to 36 of them meet with binomial weights up to 20 in one
entry (10 * 36 * 20 * 2^-24 = 4e-4)."""
import numpy as np
import pytest

from oracle import refine as OR

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # the -m gpu run happens on a GPU machine
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_13507_gb300 import refine as R  # noqa: E402


def compare(P, T, A, b, nrows, bounds, delta):
    f = lambda a: torch.tensor(a, dtype=torch.float32, device="cuda")
    h = lambda t: t.detach().double().cpu().numpy()
    P, T, A, b = f(P).requires_grad_(), f(T).requires_grad_(), f(A), f(b)
    ref = R.Refiner(P.shape[2], P.shape[2], P.shape[1] - 1, bounds, delta=delta)
    loss = R.refine_loss(P, T, A, b, torch.tensor(nrows, dtype=torch.int32, device="cuda"), ref)
    dP, dT = torch.autograd.grad(loss.sum(), (P, T))
    b32 = [float(np.float32(c)) for c in bounds]
    want = OR.loss_and_grad(h(P), h(T), h(A), h(b), nrows, b32, delta=float(np.float32(delta)))
    for got, w in zip((loss, dP, dT), want):
        assert np.all(np.abs(h(got) - w) <= 1e-3 * np.abs(w).max()), (np.abs(h(got) - w).max(), np.abs(w).max())


@pytest.mark.parametrize("m,p", [(2, 5), (3, 7)])
@pytest.mark.parametrize("c", [1e-17, 1e-18, 1e-19, 1e-20, 1e-22])
@pytest.mark.parametrize("part", [0.1, 1e-2, 1e-4])
def test_small_bounds(m, p, c, part):
    """All margins of the reach rows in the logarithm, none of the free rows."""
    rng = np.random.default_rng(3)
    S, bounds = 70, tuple(c * (k + 1) for k in range(m))
    P = rng.uniform(-1e-3, 1e-3, (S, p + 1, m)) * c
    compare(P, rng.uniform(1.0, 2.0, S), np.zeros((S, 1, m)), np.ones((S, 1)), np.zeros(S, dtype=np.int32), bounds, part * c)


@pytest.mark.parametrize("m,p", [(2, 5), (3, 7)])
@pytest.mark.parametrize("delta", [1e-18, 5e-20, 1e-20, 1e-21])
def test_small_relaxation_point(m, p, delta):
    """Free margins of delta / 2: the quadratic part, whose slope is -1.5 / delta."""
    S = 70
    A = np.zeros((S, 2, m))
    A[:, 0, 0], A[:, 1, m - 1] = 1.0, -1.0
    bounds = (2.0, 4.0) if m == 2 else (3.0, 6.0, 30.0)
    compare(np.zeros((S, p + 1, m)), np.ones(S), A, np.full((S, 2), 0.5 * delta), np.full(S, 2, dtype=np.int32), bounds, delta)
