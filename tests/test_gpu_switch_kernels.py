"""One handle switched between the kernels while it runs: the axis-chain kernel
(whose screen needs the cells' relative positions), isotropic chains, and frames
in global memory.  Positions follow the oracle through every switch.
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


@pytest.mark.parametrize("persistent", [1, 0])
def test_switching_kernels(persistent):
    N, cells, ell, nm = 1024, 6, 1.5, 2
    L = W.box_side(N, 0.66)
    x, y = W.square_lattice(N, L)
    g = P.Ecmc(N, L, 1.0, cells, cells, ell, 7)
    g.set_param(E.PARAM_N_CHAINS, nm)
    g.set_param(E.PARAM_PERSISTENT, persistent)
    axis = oracle.make_params(N, L, 1.0, cells, cells, ell, nm, 7)
    iso = oracle.make_params(N, L, 1.0, cells, cells, ell, nm, 7, dir_mode=2)
    t = 0
    for dir_mode, fmode in [(2, -1), (0, -1), (0, 2), (0, -1), (2, -1), (2, 2), (0, 1), (0, 0)]:
        g.set_param(E.PARAM_DIR_MODE, dir_mode)
        g.set_param(E.PARAM_FRAME_MODE, fmode)
        g.sweep(2)
        oracle.sweeps(iso if dir_mode else axis, x, y, t, 2)
        t += 2
        xy = g.positions()
        assert np.array_equal(xy[0::2], x) and np.array_equal(xy[1::2], y), (dir_mode, fmode)
    g.close()
