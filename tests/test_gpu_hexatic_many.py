"""The hexatic order parameter where FP64 decides many disks: a radius beyond the
FP32 decision, and crystals, whose Voronoi cells are degenerate.  On either side
of the number of disks from which a thread works on each instead of a warp; the
results are those of the oracle bit for bit.
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


@pytest.mark.parametrize("k,cells,rs,sweeps", [
    (196, 46, 3.9, 4),      # 38,416 disks, every one in FP64: a warp each
    (200, 48, 3.9, 4),      # 40,000: a thread each
    (120, 28, 3.5, 0),      # the square lattice: 14,400 undecided disks, a warp each
    (128, 30, 3.5, 0),      # 16,384: a thread each
    (128, 4, 3.5, 0),
])
def test_many_disks_in_fp64(k, cells, rs, sweeps):
    N, L = k * k, W.box_side(k * k, 0.70)
    g = P.Ecmc(N, L, 1.0, cells, cells, 1.0, 3)
    g.sweep(sweeps)
    xy = g.positions()
    x, y = np.ascontiguousarray(xy[0::2]), np.ascontiguousarray(xy[1::2])
    psi, pk, nn, bad = g.hexatic(rs=rs, per_disk=True)
    opsi, opk, onn, obad = oracle.hexatic(L, x, y, rs)
    assert bad == obad
    assert np.array_equal(nn, onn) and np.array_equal(pk, opk) and psi == opsi
    g.close()


def test_batch_with_one_crystal():
    sizes = [(10000, 0.70, 24), (16384, 0.62, 30)]
    g = P.Ecmc.batch([dict(N=n, L=W.box_side(n, eta), cells_x=c, ell=1.0, n_m=1, seed=2, replica=r)
                      for r, (n, eta, c) in enumerate(sizes)])
    g.sweep(8)
    xy = g.positions()
    lat = W.square_lattice(16384, W.box_side(16384, 0.62))
    xy[2 * 10000::2], xy[2 * 10000 + 1::2] = lat
    g.set_positions(xy, t0=8)
    psi, pk, nn, bad = g.hexatic(per_disk=True)
    off, bads = 0, 0
    for r, (n, eta, _) in enumerate(sizes):
        v = xy[2 * off:2 * (off + n)]
        opsi, opk, onn, obad = oracle.hexatic(W.box_side(n, eta), np.ascontiguousarray(v[0::2]),
                                              np.ascontiguousarray(v[1::2]))
        assert psi[r] == opsi
        assert np.array_equal(nn[off:off + n], onn) and np.array_equal(pk[off:off + n], opk)
        off, bads = off + n, bads + obad
    assert bad == bads
    g.close()
