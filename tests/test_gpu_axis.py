"""Axis chains through their static candidates (csrc/ecmc_axis.cuh): the
places where the candidates, the frame's sizes or the replay of cycles can go
wrong, against the oracle.  Trajectories are equal bit for bit, so positions
and counters are compared exactly.
"""
import math

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


def half_sigma_rows():
    # rows staggered by exactly sigma / 2: every cell of the sweeps along y
    # holds pairs on the edge between two windows, so it has no static
    # candidates
    k, L = 16, 16.4
    j, i = np.divmod(np.arange(k * k), k)
    return L, 1.02 * i + 0.5 * (j % 2), 1.025 * (j + 0.25)


def touching_columns():
    # pairs closer than sigma by 2e-10, within the overlap check, at equal
    # coordinates along x: neither is ahead of the other
    k, L = 16, 18.0
    j, i = np.divmod(np.arange(k * k), k)
    x, y = (i + 0.5) * (L / k), (j + 0.5) * (L / k)
    odd = j % 2 == 1
    y[odd] = y[~odd] + (1.0 - 2e-10)
    return L, x, y


def cluster():
    # close-packed disks in the corner of a dilute box: a few cells hold many
    # times the mean, beyond the room of a warp's cells taken together
    k, L = 16, math.sqrt(256 * math.pi / (4 * 0.05))
    j, i = np.divmod(np.arange(k * k), k)
    return L, 1.0 + (i + 0.5 * (j % 2)) * 1.003, 1.0 + j * 0.873


def melted():
    k, L = 16, W.box_side(256, 0.70)
    x, y = W.square_lattice(k * k, L)
    p = oracle.make_params(k * k, L, 1.0, 2, 2, 4.0, 2, 77)
    oracle.sweeps(p, x, y, 0, 6)
    return L, x, y


@pytest.mark.parametrize("start,cells,ell,nm", [
    (half_sigma_rows, 4, 2.0, 2),
    (half_sigma_rows, 2, 3.0, 1),   # images of the two-cell box
    (touching_columns, 4, 2.0, 2),
    (cluster, 8, 3.0, 2),
    (cluster, 4, 3.0, 17),          # more chains than start draws made at a time
    (melted, 2, 300.0, 1),          # rattles of many thousand legs, taken in whole cycles
    (melted, 6, 60.0, 1),
])
@pytest.mark.parametrize("tpc,fmode,boundary", [(1, -1, 0), (4, 0, 0), (8, 1, 0), (16, -1, 1),
                                                (32, -1, 0)])
def test_axis_chains_equal_the_oracle(start, cells, ell, nm, tpc, fmode, boundary):
    L, x, y = start()
    N = x.size
    x, y = np.mod(x, L), np.mod(y, L)
    g = P.Ecmc(N, L, 1.0, cells, cells, ell, 5)
    g.set_param(E.PARAM_N_CHAINS, nm)
    try:
        g.set_param(E.PARAM_LANES_PER_CELL, tpc)
    except E.EcmcError as e:
        assert e.code == E.ERR_UNSUPPORTED  # frames too large for so few lanes
        g.set_param(E.PARAM_LANES_PER_CELL, 0)
    g.set_param(E.PARAM_FRAME_MODE, fmode)
    g.set_param(E.PARAM_BOUNDARY, boundary)
    g.set_positions(np.stack([x, y], 1).ravel(), t0=0)
    p = oracle.make_params(N, L, 1.0, cells, cells, ell, nm, 5, boundary=boundary)
    st = oracle.Stats()
    for t in range(4):
        oracle.sweeps(p, x, y, t, 1, stats=st)
        g.sweep(1)
        xy = g.positions()
        assert np.array_equal(xy[0::2], x) and np.array_equal(xy[1::2], y), "sweep %d" % t
    c = g.counters()
    assert (c.chains, c.events, c.lifts, c.frozen_hits, c.wall_hits, c.rejected_chains) == \
        (st.chains, st.events, st.lifts, st.frozen_hits, st.wall_hits, st.rejected)
    assert c.sum_b == pytest.approx(st.sum_b, rel=1e-11, abs=1e-12)
    g.close()
