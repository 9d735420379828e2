"""A call reports its own error only: after a call has failed at its launch
(here into a capture that an earlier synchronisation made invalid), the next
call of another context succeeds."""
import ctypes

import numpy as np
import pytest

from paper_2411_13507_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # the -m gpu run happens on a GPU machine
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_13507_gb300 import plan as P  # noqa: E402


def test_a_failed_launch_is_not_reported_again():
    prob = synth.triple_integrator_3d(seed=3, N=300, K=2, nT=3)
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    one = P.Planner.for_problem(prob, arith="f32", input="f32", stream=s1)
    two = P.Planner(2, 2, 5, (2.0, 4.0), arith="f32", input="f32", stream=s2)
    dp = P.to_device(prob, input="f32")
    points = torch.rand((50, 2), device="cuda") * 20.0
    obst = P.obstacles_to_device(synth.obstacles(1, 10, 2), input="f32")
    torch.cuda.synchronize()
    graphs = one.build_batched([dp])
    outs = one.alloc_search_batched([dp])
    one.prepare_search_batched([dp], graphs, outs)
    one.search_batched_async()
    assert one.wait() == P.PLAN_OK
    two.wait()
    want = two.obstacle_planes(points, obst)
    got = {k: torch.zeros_like(v) for k, v in want.items()}
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    stream, graph = ctypes.c_void_p(s1.cuda_stream), ctypes.c_void_p()
    assert cu.cuStreamBeginCapture_v2(stream, 2) == 0  # relaxed: other streams are free to work
    try:
        assert one.lib.plan_wait(one.ctx, None) == P.PLAN_ERR_CUDA  # not allowed in a capture, which ends it
        with pytest.raises(P.PlanError):
            one.search_batched_async()
        two.obstacle_planes_async(points, obst, got)
    finally:
        cu.cuStreamEndCapture(stream, ctypes.byref(graph))
    assert two.wait() == P.PLAN_OK
    for k in want:
        assert np.array_equal(got[k].cpu().numpy(), want[k].cpu().numpy())
