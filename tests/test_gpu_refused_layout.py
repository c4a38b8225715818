"""A parameter that the handle refuses leaves it as it was: the launch shape,
its buffers and the parameters read back, so that the next sweep continues the
oracle's trajectory.
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

KEYS = (E.PARAM_LANES_PER_CELL, E.PARAM_FRAME_MODE, E.PARAM_PERSISTENT, E.PARAM_DIR_MODE,
        E.PARAM_BOUNDARY, E.PARAM_WARPS_PER_BLOCK, E.PARAM_STRIP_WIDTH, E.PARAM_KERNELS_PER_SWEEP)


@pytest.mark.parametrize("persistent", [1, 0])
@pytest.mark.parametrize("kind", ["axis", "rejecting", "isotropic"])
@pytest.mark.parametrize("graph", [1, 0])
def test_sweep_after_refused_lanes(kind, persistent, graph):
    # 33-sigma cells: frames for 16 cells a warp fit nowhere
    N, eta, cells, ell, nm = 4096, 0.72, 2, 0.2 if kind == "rejecting" else 3.0, 3
    L = W.box_side(N, eta)
    x, y = W.square_lattice(N, L)
    g = P.Ecmc(N, L, 1.0, cells, cells, ell, 7)
    g.set_param(E.PARAM_N_CHAINS, nm)
    g.set_param(E.PARAM_PERSISTENT, persistent)
    g.set_param(E.PARAM_USE_GRAPH, graph)
    p = oracle.make_params(N, L, 1.0, cells, cells, ell, nm, 7)
    if kind == "rejecting":
        g.set_param(E.PARAM_BOUNDARY, E.BOUNDARY_REJECT)
        p = oracle.make_params(N, L, 1.0, cells, cells, ell, nm, 7, boundary=1)
    elif kind == "isotropic":
        g.set_param(E.PARAM_DIR_MODE, E.DIR_ISOTROPIC)
        p = oracle.make_params(N, L, 1.0, cells, cells, ell, nm, 7, dir_mode=2)
    g.sweep(1)
    before = [g.get_param(k) for k in KEYS]
    for lanes in (2, 1):
        with pytest.raises(E.EcmcError) as ei:
            g.set_param(E.PARAM_LANES_PER_CELL, lanes)
        assert ei.value.code == E.ERR_UNSUPPORTED and "%d lanes" % lanes in str(ei.value)
        assert [g.get_param(k) for k in KEYS] == before
    g.sweep(2)
    oracle.sweeps(p, x, y, 0, 3)
    xy = g.positions()
    if kind == "isotropic":
        assert np.abs(xy[0::2] - x).max() < 1e-9 and np.abs(xy[1::2] - y).max() < 1e-9
    else:
        assert np.array_equal(xy[0::2], x) and np.array_equal(xy[1::2], y)
    g.close()
