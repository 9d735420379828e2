"""The screened pair kernel (k_pairs_sc) where its FP16 rows and its box rows
can go wrong: durations so short that the rows leave the FP16 range, states so
close together that FP16 decides few pairs, polytopes with scaled, repeated,
missing, zero and redundant rows along the axes, tiles of one pair up to just
above a full one, and enough feasible pairs for staged costs beside too few.
Graphs equal the FP64 oracle's (masks and edges exactly, weights within 1e-5).
"""
import numpy as np
import pytest

import oracle
from paper_2411_13507_gb300 import synth

KHF = 17 / 16 * 2.0 ** -10
EH = 2.0 ** -20


def test_fp16_row_band_covers_the_rounding():
    """The FP16 sum of two rounded halves stays within KHF (|u| + |w|) + EH of their exact sum."""
    from test_screen_fp16_bound import fp16_sum, samples
    u, w = samples(400_000, 23)
    mag = np.abs(u.astype(np.float64)) + np.abs(w.astype(np.float64))
    err = np.abs(fp16_sum(u, w) - (u.astype(np.float64) + w.astype(np.float64)))
    assert np.all(err <= KHF * mag + EH)


def build(prob, **kw):
    from paper_2411_13507_gb300 import plan as P
    pl = P.Planner.for_problem(prob, arith="f32")
    pl.set_tile(**kw)
    g = pl.build_edges(P.to_device(prob, input=prob.dtype)).to_numpy()
    pl.close()
    return g


def check(prob, **kw):
    import parity
    g = build(prob, **kw)
    csr = oracle.OracleProblem(prob).csr(with_detail=True)
    parity.compare_full(g, csr, prob.N, prob.nT, "f32")
    return g


def environment(seed, m, p, N, K, T, spread=None):
    f = synth.double_integrator_2d if m == 2 else synth.triple_integrator_3d
    prob = f(seed, N=N, K=K, nT=len(T), degree=p)
    prob.T = np.asarray(np.asarray(T, dtype=np.float32), dtype=np.float64)
    if spread is not None:  # every state near one point of the first polytope, and slow
        rng = np.random.default_rng(seed)
        prob.states[:, :m] = prob.states[0, :m] + rng.uniform(-spread, spread, (N, m))
        prob.states[:, m:] *= spread
        prob.states = prob.states.astype(np.float32).astype(np.float64)
    return prob


@pytest.mark.gpu
@pytest.mark.parametrize("m,p", [(2, 3), (2, 5), (3, 5), (3, 7)])
@pytest.mark.parametrize("N,K", [(2, 1), (9, 1), (65, 1), (150, 2)])
def test_sizes_and_short_durations(m, p, N, K):
    check(environment(3, m, p, N, K, [0.004, 0.03, 0.2, 0.7, 1.5, 2.6]))


@pytest.mark.gpu
@pytest.mark.parametrize("m,p", [(2, 5), (3, 5), (3, 7)])
@pytest.mark.parametrize("spread", [1e-5, 1e-3, 0.03])
def test_states_close_together(m, p, spread):
    check(environment(5, m, p, 70, 1, [0.02, 0.1, 0.5, 2.0], spread))


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["scaled", "repeated", "none", "zero", "tiny"])
@pytest.mark.parametrize("m,p", [(2, 5), (3, 7)])
def test_polytope_rows(kind, m, p):
    prob = environment(7, m, p, 120, 2, [0.4, 0.9, 1.6, 2.4])
    rows = [(prob.A[a:b].copy(), prob.b[a:b].copy()) for a, b in zip(prob.poly_off[:-1], prob.poly_off[1:])]
    out = []
    for A, b in rows:
        if kind == "scaled":      # rows of other lengths, one 2^20 times another
            s = 2.0 ** np.linspace(-8, 12, len(b)).round()
            A, b = A * s[:, None], b * s
        elif kind == "repeated":  # several rows along the same axis and sign, the later ones tighter
            A, b = np.concatenate([A, A[:2 * m]]), np.concatenate([b, b[:2 * m] - 0.05 * np.abs(b[:2 * m])])
        elif kind == "none":      # no row along an axis: a turned box
            c, s = np.cos(0.3), np.sin(0.3)
            Rm = np.eye(m)
            Rm[:2, :2] = [[c, -s], [s, c]]
            if m == 3:
                Rm = Rm @ np.array([[c, 0, -s], [0, 1, 0], [s, 0, c]])
            ctr = prob.states[0, :m]
            A = np.concatenate([Rm, -Rm])
            b = A @ ctr + 2.0
        elif kind == "zero":      # a row without a normal
            A, b = np.concatenate([A, np.zeros((1, m))]), np.concatenate([b, [1.0]])
        else:                     # an axis row with a second entry far below the first
            A = A.copy()
            A[0, 1] = 1e-30
        out.append((A, b))
    prob.poly_off = np.concatenate([[0], np.cumsum([len(b) for _, b in out])]).astype(np.int32)
    prob.A = np.concatenate([A for A, _ in out]).astype(np.float32).astype(np.float64)
    prob.b = np.concatenate([b for _, b in out]).astype(np.float32).astype(np.float64)
    check(prob)


@pytest.mark.gpu
@pytest.mark.parametrize("tile", [8, 20, 64])
@pytest.mark.parametrize("cost", ["state", "pos"])
def test_tiles_and_cost_rows(tile, cost):
    prob = environment(11, 3, 7, 300, 3, [0.3, 1.2, 2.0, 2.8])
    prob.model.cost_mode = cost
    check(prob, tile=tile, tchunks=1)
    check(prob, tile=tile, tchunks=4)
