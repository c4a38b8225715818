"""The count of candidates evaluated in FP64 by axis chains with static
candidates: three for every leg; in a cell without static candidates, where
each leg searches the whole frame, every other object as well.
"""
import numpy as np
import pytest

import ecmc_workloads as W
import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1409_6948_gb300 as P  # noqa: E402
from paper_1409_6948_gb300 import ecmc as E  # noqa: E402


def frame_objects(p, t, x, y):
    """Members and images within sigma of each cell of sweep t."""
    sx, sy, _ = oracle.sweep_draws(p, t)
    w, out = p.L / p.cells_x, []
    for cy in range(p.cells_y):
        for cx in range(p.cells_x):
            nx = np.zeros(x.size, int)
            ny = np.zeros(x.size, int)
            for m in (-1, 0, 1):
                X = np.mod(x - (sx + cx * w) + 0.5 * p.L, p.L) - 0.5 * p.L + m * p.L
                Y = np.mod(y - (sy + cy * w) + 0.5 * p.L, p.L) - 0.5 * p.L + m * p.L
                nx += (X > -1.0) & (X < w + 1.0)
                ny += (Y > -1.0) & (Y < w + 1.0)
            out.append(int(np.sum(nx * ny)))
    return out


@pytest.mark.parametrize("lanes", [2, 8, 32])
@pytest.mark.parametrize("cells", [4, 2])
def test_one_leg_per_chain(lanes, cells):
    # ell = 0: every chain is one leg and nothing moves.  Rows staggered by
    # sigma / 2: no cell of a sweep along y has static candidates
    k, L, nm = 16, 16.4, 5
    j, i = np.divmod(np.arange(k * k), k)
    x, y = np.mod(1.02 * i + 0.5 * (j % 2), L), np.mod(1.025 * (j + 0.25), L)
    g = P.Ecmc(k * k, L, 1.0, cells, cells, 0.0, 5)
    g.set_param(E.PARAM_N_CHAINS, nm)
    g.set_param(E.PARAM_LANES_PER_CELL, lanes)
    g.set_positions(np.stack([x, y], 1).ravel(), t0=0)
    p = oracle.make_params(k * k, L, 1.0, cells, cells, 0.0, nm, 5)
    want = 0
    for t in range(4):
        g.sweep(1)
        if t % 2 == 0:
            want += 3 * nm * cells * cells
        else:
            want += nm * sum(2 + n for n in frame_objects(p, t, x, y))
        assert g.counters().fp64_evals == want, t
    g.close()


def test_legs_of_moving_chains():
    # regular cells, no replay: three for every event, reflection and chain end
    N, L = 4096, W.box_side(4096, 0.70)
    g = P.Ecmc(N, L, 1.0, 16, 16, 2.0, 5)
    g.set_param(E.PARAM_REPLAY, 0)
    g.sweep(3)
    g.reset_stats()
    g.sweep(3)
    c = g.counters()
    legs = c.events + c.wall_hits + c.chains
    assert c.replayed_legs == 0 and c.fp64_evals >= 3 * legs
    assert c.fp64_evals <= 3 * legs + 0.01 * legs * 60  # (a stray irregular cell)
    g.close()


@pytest.mark.parametrize("boundary,persistent", [(0, 1), (0, 0), (1, 1)])
def test_only_the_pair_on_an_edge_searches(boundary, persistent):
    # one pair of a melted configuration exactly sigma / 2 apart across the
    # axis: the legs of these two search their frame, those of the cell's other
    # 670 members do not
    N, cells, (nm, ell) = 2704, 2, ((30, 3.0) if boundary == 0 else (60, 0.4))
    L = W.box_side(N, 0.72)
    p = oracle.make_params(N, L, 1.0, cells, cells, ell, nm, 5, boundary=boundary)
    x, y = W.square_lattice(N, L)
    oracle.sweeps(oracle.make_params(N, L, 1.0, 12, 12, 2.0, 10, 6), x, y, 0, 60)
    sx, _, _ = oracle.sweep_draws(p, 1)
    w, done = L / cells, 0
    for o in range(N):
        u = np.mod(x - sx, L)
        near = np.nonzero((np.abs(np.abs(x - x[o]) - 0.5) < 2e-3) & (u // w == u[o] // w)
                          & (np.abs(y - y[o]) < 6.0))[0]
        for j in near:
            old = x[o]
            x[o] = x[j] + np.copysign(0.5, old - x[j])
            if 0 < x[o] < L and oracle.min_dist2(L, x, y) > 1.0 - 1e-10:
                done += 1
                break
            x[o] = old
        if done:
            break
    assert done
    g = P.Ecmc(N, L, 1.0, cells, cells, ell, 5)
    g.set_param(E.PARAM_N_CHAINS, nm)
    g.set_param(E.PARAM_BOUNDARY, boundary)
    g.set_param(E.PARAM_PERSISTENT, persistent)
    assert g.get_param(E.PARAM_KERNELS_PER_SWEEP) == (5 if persistent else 8)
    g.set_positions(np.stack([x, y], 1).ravel(), t0=1)
    g.sweep(1)
    oracle.sweeps(p, x, y, 1, 1)
    xy = g.positions()
    assert np.array_equal(xy[0::2], x) and np.array_equal(xy[1::2], y)
    c = g.counters()
    legs = c.events + c.wall_hits + c.chains - c.replayed_legs - c.rejected_chains
    assert 3 * legs <= c.fp64_evals < 3 * legs + 0.03 * legs * 800
    g.close()
