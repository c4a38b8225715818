"""Which kernel runs axis chains in large cells, and that each follows the oracle:
the kernel of static candidates where a cell's chains are long enough to pay for
them, the per-phase kernels otherwise, where FP32 is too coarse for the
candidates (38 sigma and more at fluid density) and where frames do not fit.
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


def compare(g, x, y, st):
    xy = g.positions()
    assert np.array_equal(xy[0::2], x) and np.array_equal(xy[1::2], y)
    c = g.counters()
    assert (c.events, c.lifts, c.frozen_hits, c.wall_hits) == \
        (st.events, st.lifts, st.frozen_hits, st.wall_hits)


# about 49 legs a chain; static candidates pay from 49, 117, 308 and 462 legs a cell
# of 16.7, 20.9, 27.1 and 31.3 sigma, from 389 at 27.1 sigma under ECMC_PREC_FP64
@pytest.mark.parametrize("k,side,nm,prec,persistent,fmode,kernels", [
    (32, 16.7, 2, 1, 1, -1, 5),
    (40, 20.9, 1, 1, 1, -1, 12),
    (40, 20.9, 4, 1, 1, -1, 5),
    (52, 27.1, 8, 1, 1, -1, 5),
    (52, 27.1, 8, 1, 0, -1, 8),
    (52, 27.1, 8, 1, 1, 0, 5),       # candidate lists in shared memory
    (52, 27.1, 4, 1, 1, -1, 12),
    (52, 27.1, 8, 0, 1, -1, 5),
    (52, 27.1, 6, 0, 1, -1, 12),
    (60, 31.3, 16, 1, 1, -1, 5),
    (60, 31.3, 16, 1, 1, 0, 12),     # no room for the lists in shared memory
    (72, 37.6, 40, 1, 1, -1, 12),    # FP32 too coarse
    (76, 39.7, 40, 1, 1, 1, 12),
    (88, 46.0, 6, 0, 1, -1, 12),
    (96, 50.1, 6, 1, 1, -1, 12),     # frames beyond the kernel's shared memory
    (96, 50.1, 6, 1, 0, 1, 12),
])
def test_kernel_of_large_cells(k, side, nm, prec, persistent, fmode, kernels):
    N, L, ell = k * k, W.box_side(k * k, 0.72), 3.0
    assert abs(L / 2 - side) < 0.1
    x, y = W.square_lattice(N, L)
    g = P.Ecmc(N, L, 1.0, 2, 2, ell, 5)
    g.set_param(E.PARAM_N_CHAINS, nm)
    g.set_param(E.PARAM_PRECISION, prec)
    g.set_param(E.PARAM_PERSISTENT, persistent)
    g.set_param(E.PARAM_FRAME_MODE, fmode)
    assert g.get_param(E.PARAM_KERNELS_PER_SWEEP) == kernels
    p = oracle.make_params(N, L, 1.0, 2, 2, ell, nm, 5)
    st, _ = oracle.sweeps(p, x, y, 0, 6)
    g.sweep(6)
    compare(g, x, y, st)
    g.close()


def test_chains_per_cell_switch_the_kernel():
    # the number of chains changes between sweeps, and the kernel with it
    N, L, ell = 2704, W.box_side(2704, 0.72), 3.0
    x, y = W.square_lattice(N, L)
    g = P.Ecmc(N, L, 1.0, 2, 2, ell, 5)
    t, st = 0, oracle.Stats()
    for nm, kernels in [(1, 12), (9, 5), (2, 12), (12, 5)]:
        g.set_param(E.PARAM_N_CHAINS, nm)
        assert g.get_param(E.PARAM_KERNELS_PER_SWEEP) == kernels
        g.sweep(2)
        p = oracle.make_params(N, L, 1.0, 2, 2, ell, nm, 5)
        oracle.sweeps(p, x, y, t, 2, stats=st)
        t += 2
        compare(g, x, y, st)
    g.close()
