"""Measurements where their kernels take another path: the hexatic order
parameter's FP32 decision and its FP64 remainder, several warps per cell, and
the overlap check of a batch whose replicas need different scans.  Results are
those of the oracle bit for bit.
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


@pytest.mark.parametrize("N,eta,cells,rs", [
    (1024, 0.70, 8, 2.5),
    (1024, 0.70, 4, 3.5),    # 64 members per cell: two chunks of lanes
    (1024, 0.70, 8, 3.9),    # beyond the packing bound of the 64-disk limit: FP64 only
    (900, 0.30, 6, 3.5),     # dilute: open and uncertified cells go to FP64
    (64, 0.66, 2, 3.5),      # a disk's images across the box
])
def test_hexatic_paths_bitwise(N, eta, cells, rs):
    L = W.box_side(N, eta)
    g = P.Ecmc(N, L, 1.0, cells, cells, 2.0, 3)
    g.sweep(40)
    xy = g.positions()
    x, y = np.ascontiguousarray(xy[0::2]), np.ascontiguousarray(xy[1::2])
    psi, pk, nn, bad = g.hexatic(rs=rs, per_disk=True)
    opsi, opk, onn, obad = oracle.hexatic(L, x, y, rs)
    assert bad == obad
    assert np.array_equal(nn, onn) and np.array_equal(pk, opk) and psi == opsi
    g.close()


def test_overlap_check_of_a_mixed_batch():
    # a box below 8 sigma (FP64 scan), one with the full stencil, one with the
    # half stencil and two warps per cell
    sizes = [(36, 0.60, 2), (256, 0.70, 2), (4096, 0.70, 8)]
    descs = [dict(N=N, L=W.box_side(N, eta), cells_x=c, ell=1.0, n_m=2, seed=4, replica=r)
             for r, (N, eta, c) in enumerate(sizes)]
    g = P.Ecmc.batch(descs)
    g.sweep(12)
    xy, off, least = g.positions(), 0, []
    for d in descs:
        v = xy[2 * off:2 * (off + d["N"])]
        least.append(oracle.min_dist2(d["L"], np.ascontiguousarray(v[0::2]),
                                      np.ascontiguousarray(v[1::2])))
        off += d["N"]
    assert g.min_distance() == math.sqrt(min(least))
    g.close()
