"""plan_mpc_qp in captured graphs beside direct calls of the same context: each
replay and each direct call solves the problems of its own parameters, whatever
horizons and weights ran in between.  The kernel is deterministic, so every
result equals a fresh context's bit for bit."""
import numpy as np
import pytest

from mpc_cases import instance

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # the -m gpu run happens on a GPU machine
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_13507_gb300 import plan as P  # noqa: E402


class Case:
    """Four problems of one horizon and one set of weights, and their solution by a fresh context."""

    def __init__(self, H, q=1.0, seed=1):
        insts = [instance(seed + i, H=H) for i in range(4)]
        self.H, self.q, self.i0 = H, q, insts[0]
        t = lambda k, dt: torch.tensor(np.stack([i[k] for i in insts]), dtype=dt, device="cuda")
        self.x0, self.ref, self.planes = t("x0", torch.float64), t("ref", torch.float64), t("planes", torch.float32)
        pl = self.planner(torch.cuda.Stream())
        out = self.call(pl)
        assert pl.wait() == P.PLAN_OK
        self.want = {k: v.cpu().numpy() for k, v in out.items()}
        assert np.all(self.want["status"] == P.PLAN_MPC_OK)

    def planner(self, stream):
        torch.cuda.synchronize()
        return P.Planner(2, 2, 5, self.i0["bounds"], arith="f64", input="f64", stream=stream)

    def call(self, pl, out=None):
        i = self.i0
        prm = pl.mpc_params(self.H, i["dt"], self.q * i["Q"], i["F"], i["R"], i["V"])
        out = pl.alloc_mpc(4, self.H) if out is None else out
        torch.cuda.current_stream().synchronize()
        pl.mpc_qp_async(prm, self.x0, self.ref, self.planes, out)
        return out

    def capture(self, pl):
        i = self.i0
        prm, out = pl.mpc_params(self.H, i["dt"], self.q * i["Q"], i["F"], i["R"], i["V"]), pl.alloc_mpc(4, self.H)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=pl.stream):
            pl.mpc_qp_async(prm, self.x0, self.ref, self.planes, out)
        return g, out

    def replay(self, pl, captured):
        g, out = captured
        for v in out.values():
            v.zero_()
        torch.cuda.synchronize()
        with torch.cuda.stream(pl.stream):
            g.replay()
        pl.stream.synchronize()
        self.check(out)

    def check(self, out):
        assert all(np.array_equal(out[k].cpu().numpy(), self.want[k]) for k in self.want)

    def direct(self, pl):
        out = self.call(pl)
        assert pl.wait() == P.PLAN_OK
        self.check(out)


def test_a_replay_between_equal_direct_calls():
    a, b = Case(10), Case(5)
    pl = a.planner(torch.cuda.Stream())
    a.direct(pl)
    g = b.capture(pl)
    a.direct(pl)
    b.replay(pl, g)
    a.direct(pl)
    b.replay(pl, g)
    a.direct(pl)


def test_first_call_captured_and_larger_calls_after_it():
    a, b, c = Case(5), Case(8, q=3.0), Case(20)
    pl = a.planner(torch.cuda.Stream())
    ga = a.capture(pl)
    c.direct(pl)          # grows the direct calls' buffers
    gb = b.capture(pl)
    gc = c.capture(pl)
    for x, g in ((a, ga), (b, gb), (c, gc), (b, gb), (a, ga)):
        x.replay(pl, g)
        c.direct(pl)


def test_same_parameters_captured_twice():
    a = Case(7)
    pl = a.planner(torch.cuda.Stream())
    g1, g2 = a.capture(pl), a.capture(pl)
    a.replay(pl, g1)
    a.direct(pl)
    a.replay(pl, g2)
    a.replay(pl, g1)
