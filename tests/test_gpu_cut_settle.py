"""Cut entries that only FP64 settles, many to a block of the pair kernel: curves
along one line over obstacle corners that miss or reach it by a few 1e-7 (inside
the FP32 bands, far outside FP64 rounding), for obstacles of 3, 8, 9 and 16
rows.  Kept edges and masks bit-exact against the oracle, no tie."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # the -m gpu run happens on a GPU machine
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2411_13507_gb300 import synth  # noqa: E402
from test_gpu_cut import check  # noqa: E402


def line_problem():
    """States at rest on both sides of x = 2 on the line y = 2: every curve is a segment of it."""
    prob, _ = synth.keepout_2d(11, N=48, n_obst=1, width=4.0)
    rng = np.random.default_rng(7)
    prob.states[:, :] = 0.0
    prob.states[:24, 0] = rng.uniform(0.6, 1.6, 24)
    prob.states[24:, 0] = rng.uniform(2.4, 3.4, 24)
    prob.states[:, 1] = 2.0
    prob.model.bounds = (50.0, 500.0)
    return prob


def corners(rows, n=12):
    """n polygons below the line, one corner up at y = 2 + d, d = +-1e-7 .. +-6e-7."""
    off, A, b = [0], [], []
    for k in range(n):
        d = (1 + k // 2) * (1e-7 if k % 2 else -1e-7)
        top = np.array([1.7 + 0.6 * (k + 0.5) / n, 2.0 + d])
        if rows == 3:
            nrm = np.array([[np.sqrt(0.5), np.sqrt(0.5)], [-np.sqrt(0.5), np.sqrt(0.5)], [0.0, -1.0]])
            rhs = nrm @ top + np.array([0.0, 0.0, 0.2])
        else:  # regular polygon of radius R with a vertex at the top
            R = 0.1
            th = np.pi / 2 + 2 * np.pi * (np.arange(rows) + 0.5) / rows
            nrm = np.stack([np.cos(th), np.sin(th)], axis=1)
            rhs = nrm @ (top - np.array([0.0, R])) + R * np.cos(np.pi / rows)
            up = nrm @ top - rhs            # the two facets of the top vertex go through it exactly
            rhs = np.where(np.abs(up) < 1e-9, nrm @ top, rhs)
        A.append(nrm)
        b.append(rhs)
        off.append(off[-1] + rows)
    return synth.Obstacles(np.array(off, dtype=np.int32), np.concatenate(A), np.concatenate(b))


@pytest.mark.parametrize("rows", [3, 8, 9, 16])
def test_many_entries_settled_in_fp64(rows):
    st, info, orc, gpu, g, out = check(line_problem(), corners(rows), "f64")
    assert info["cut_lp64"] > 1000
