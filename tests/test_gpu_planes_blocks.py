"""All-pairs closest points in 2-D by blocks of obstacles: counts around whole
warps and blocks, few points, many rows, outputs at odd addresses.  A call with
all obstacles must equal, bit for bit, calls with 20 of them at a time (which
take the kernel that reads the geometry per pair)."""
import numpy as np
import pytest

from paper_2411_13507_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # the -m gpu run happens on a GPU machine
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_13507_gb300 import plan as P  # noqa: E402


def part(obs, a, b):
    r0, r1 = obs.off[a], obs.off[b]
    return synth.Obstacles(obs.off[a:b + 1] - r0, obs.A[r0:r1], obs.b[r0:r1])


def call(pl, pts, do, shift=0):
    n, m = do.n, pts.shape[0]
    new = lambda k, dt=torch.float32: torch.full((k + shift,), -7, dtype=dt, device="cuda")[shift:]
    out = {"closest": new(m * n * 2), "plane": new(m * n * 3), "dist": new(m * n),
           "nearest": new(m, torch.int32), "nearest_dist": new(m)}
    pl.obstacle_planes_async(pts, do, out)
    assert pl.wait() == P.PLAN_OK
    return {k: v.clone() for k, v in out.items()}


@pytest.mark.parametrize("n,points", [(23, 9), (24, 1), (31, 5), (32, 12), (33, 2), (96, 7), (127, 13), (128, 50), (129, 3),
                                      (300, 200)])
@pytest.mark.parametrize("cuts,input,shift", [(3, "f32", 0), (3, "f64", 1), (12, "f32", 0)])
def test_blocks_equal_single_pairs(n, points, cuts, input, shift):
    obs = synth.obstacles(n, n, 2, domain=(0.0, 3.0), side=(0.05, 0.6), max_cuts=cuts, dtype=input)
    pl = P.Planner(2, 2, 5, (2.0, 4.0), arith=input, input=input)
    pts = torch.tensor(np.random.default_rng(n).uniform(0, 3, (points, 2)), device="cuda",
                       dtype=torch.float32 if input == "f32" else torch.float64)
    got = call(pl, pts, P.obstacles_to_device(obs, input), shift)
    refs = [call(pl, pts, P.obstacles_to_device(part(obs, a, min(n, a + 20)), input)) for a in range(0, n, 20)]
    for k, w in (("closest", 2), ("plane", 3), ("dist", 1)):
        ref = torch.cat([r[k].view(points, -1, w) for r in refs], 1)
        assert torch.equal(got[k].view(points, n, w), ref), k
    d = got["dist"].view(points, n)
    assert torch.equal(got["nearest_dist"], d.min(1).values)
    assert torch.equal(got["nearest"].long(), (d == d.min(1, keepdim=True).values).float().argmax(1))
