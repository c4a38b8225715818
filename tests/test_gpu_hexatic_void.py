"""The hexatic order parameter where a disk stands alone: its Delaunay
neighbours lie beyond the candidates of the FP32 decision (2.2 mean spacings),
so the FP64 decision over all disks within rs has to take it.  Results are those
of the oracle bit for bit, the count of uncertified disks included.
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


def strip_with_a_lone_disk(gap):
    # 17 staggered rows of 19 disks, an empty strip of width `gap` between the
    # last and the first, one disk in its middle
    L, cols, rows = 20.4, 19, 17
    a, h = L / cols, (L - gap) / (rows - 1)
    j, i = np.divmod(np.arange(cols * rows), cols)
    x, y = (i + 0.5 * (j % 2)) * a, 0.5 + j * h
    x = np.append(x, 0.3 * L)
    y = np.append(y, 0.5 + (rows - 1) * h + 0.5 * gap)
    return L, np.mod(x, L), np.mod(y, L)


# nearest disks at 3.0 to 3.35 sigma, candidates within 2.49: neighbours in rs,
# or none there either
@pytest.mark.parametrize("gap", [6.0, 6.27, 6.7])
@pytest.mark.parametrize("rs", [3.5, 2.6, 2.0])
@pytest.mark.parametrize("cells", [2, 4])
def test_disk_without_candidates(gap, rs, cells):
    L, x, y = strip_with_a_lone_disk(gap)
    g = P.Ecmc(x.size, L, 1.0, cells, cells, 1.0, 3)
    g.set_positions(np.stack([x, y], 1).ravel(), t0=0)
    psi, pk, nn, bad = g.hexatic(rs=rs, per_disk=True)
    opsi, opk, onn, obad = oracle.hexatic(L, x, y, rs)
    assert bad == obad
    assert np.array_equal(nn, onn) and np.array_equal(pk, opk) and psi == opsi
    g.close()


def test_one_replica_of_a_batch_has_a_void():
    L, x, y = strip_with_a_lone_disk(6.27)
    sizes = [(1024, W.box_side(1024, 0.70), 8), (x.size, L, 4)]
    g = P.Ecmc.batch([dict(N=n, L=side, cells_x=c, ell=1.0, n_m=1, seed=2, replica=r)
                      for r, (n, side, c) in enumerate(sizes)])
    g.sweep(10)
    xy = g.positions()
    xy[2 * 1024::2], xy[2 * 1024 + 1::2] = x, y
    g.set_positions(xy, t0=10)
    psi, pk, nn, bad = g.hexatic(per_disk=True)
    off, bads = 0, 0
    for r, (n, side, _) in enumerate(sizes):
        v = xy[2 * off:2 * (off + n)]
        opsi, opk, onn, obad = oracle.hexatic(side, np.ascontiguousarray(v[0::2]),
                                              np.ascontiguousarray(v[1::2]))
        assert np.array_equal(nn[off:off + n], onn) and np.array_equal(pk[off:off + n], opk)
        assert psi[r] == opsi
        off, bads = off + n, bads + obad
    assert bad == bads
    g.close()
