"""Refinement loss and gradients where a block of segments or a chunk of staged
polytope rows ends: one segment, a block less and more one, no row, rows past a
chunk.  Against the FP64 oracle, segment by segment: within 3e-5 of the
output's largest value (a sum of up to 500 FP32 terms, 500 * 2^-24), the
loss's logarithms, of either sign, counted with one each."""
import numpy as np
import pytest

from oracle import refine as OR
from paper_2411_13507_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # the -m gpu run happens on a GPU machine
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_13507_gb300 import refine as R  # noqa: E402


@pytest.mark.parametrize("m,p", [(2, 5), (3, 7)])
@pytest.mark.parametrize("S,rmax", [(1, 12), (63, 12), (64, 12), (65, 12), (70, 0), (5, 6), (130, 16), (67, 17), (3, 33), (66, 64)])
def test_against_the_oracle(m, p, S, rmax):
    bounds = (2.0, 4.0) if m == 2 else (3.0, 6.0, 30.0)
    full = max(rmax, 2 * m)
    rb = synth.refine_segments(seed=S, S=S, degree=p, m=m, rmax=full, max_cuts=full - 2 * m, bounds=bounds)
    rb.nrows = np.minimum(rb.nrows, rmax)
    f = lambda a: torch.tensor(np.asarray(a), dtype=torch.float32, device="cuda")
    P, T, A, b = f(rb.P), f(rb.T), f(rb.A)[:, :rmax].contiguous(), f(rb.b)[:, :rmax].contiguous()
    nrows = torch.tensor(rb.nrows, dtype=torch.int32, device="cuda")
    up = torch.linspace(0.5, 2.0, S, device="cuda")
    ref = R.Refiner(m, m, p, bounds)
    P.requires_grad_()
    T.requires_grad_()
    loss = R.refine_loss(P, T, A, b, nrows, ref)
    dP, dT = torch.autograd.grad(loss, (P, T), up)
    h = lambda t: t.detach().double().cpu().numpy()
    lo, dPo, dTo = OR.loss_and_grad(h(P), h(T), h(A), h(b), rb.nrows, bounds)
    w = h(up)
    for got, want in ((h(loss), lo), (h(dP), dPo * w[:, None, None]), (h(dT), dTo * w)):
        scale = np.abs(want).reshape(S, -1).max(1).reshape((S,) + (1,) * (want.ndim - 1)) + 500.0
        assert np.all(np.abs(got - want) <= 3e-5 * scale)
