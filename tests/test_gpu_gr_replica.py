"""g(r) of one replica of an uneven batch, measured by itself: only its own cells
are converted to fixed point, and the counts are the oracle's integers.
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


@pytest.mark.parametrize("order", [(0, 1, 2, 3), (3, 1), (2,)])
def test_single_replicas(order):
    # the second takes the FP64 scan (rmax beyond a quarter of its box)
    sizes = [(1024, 0.70, 8), (256, 0.66, 2), (4096, 0.72, 16), (1600, 0.60, 10)]
    descs = [dict(N=n, L=W.box_side(n, eta), cells_x=c, ell=2.0, n_m=2, seed=4, replica=r)
             for r, (n, eta, c) in enumerate(sizes)]
    g = P.Ecmc.batch(descs)
    g.set_param(E.PARAM_GR_DR, 0.02)
    g.set_param(E.PARAM_GR_RMAX, 5.0)
    g.sweep(6)
    xy = g.positions()
    off = np.concatenate([[0], np.cumsum([d["N"] for d in descs])])
    for r in order:
        g.gr_measure(r)
    for r, d in enumerate(descs):
        v = xy[2 * off[r]:2 * off[r + 1]]
        got, n_meas = g.gr_counts(r)
        want = oracle.gr_counts(d["L"], np.ascontiguousarray(v[0::2]),
                                np.ascontiguousarray(v[1::2]), 1.0, 0.02, 200)
        assert n_meas == (1 if r in order else 0)
        assert np.array_equal(got, want if r in order else 0 * want), r
    g.close()
