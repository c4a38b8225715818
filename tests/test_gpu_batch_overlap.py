"""The overlap check of a batch whose replicas have disks of different sizes:
each replica's smallest distance counts against its own diameter.
"""
import numpy as np
import pytest

import ecmc_workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

import paper_1409_6948_gb300 as P  # noqa: E402
from paper_1409_6948_gb300 import ecmc as E  # noqa: E402

# (N, cells, sigma): boxes below 8 sigma (FP64 scan), the full and the half
# stencil of the fixed-point scan
SIZES = [(36, 2, 1.0), (256, 2, 2.0), (4096, 8, 0.5), (1024, 4, 2.0), (36, 2, 3.0)]


def batch():
    descs = [dict(N=n, L=W.box_side(n, 0.60) * s, sigma=s, cells_x=c, ell=0.5 * s, n_m=1,
                  seed=1, replica=r) for r, (n, c, s) in enumerate(SIZES)]
    return P.Ecmc.batch(descs), descs


def lattices(descs):
    return [W.square_lattice(d["N"], d["L"]) for d in descs]


def joined(parts):
    return np.concatenate([np.stack(p, 1).ravel() for p in parts])


@pytest.mark.parametrize("replica", range(len(SIZES)))
@pytest.mark.parametrize("distance,overlaps", [(0.75, True), (1.0 - 1e-8, True),
                                               (1.0 - 1e-10, False), (1.0 + 1e-8, False)])
def test_each_replica_against_its_own_diameter(replica, distance, overlaps):
    g, descs = batch()
    parts = lattices(descs)
    # disk 1 moves towards disk 0 along x
    x, y = parts[replica]
    x[1] = x[0] + distance * descs[replica]["sigma"]
    xy = joined(parts)
    if overlaps:
        with pytest.raises(E.EcmcError) as ei:
            g.set_positions(xy, t0=0)
        assert ei.value.code == E.ERR_OVERLAP
        with pytest.raises(E.EcmcError) as ei:
            g.sweep(1)
        assert ei.value.code == E.ERR_STATE
        g.set_positions(joined(lattices(descs)), t0=0)
    else:
        g.set_positions(xy, t0=0)
    # the smallest distance of all replicas, whatever their diameters (pairs
    # within two diameters of their replica)
    least = min(np.hypot(np.diff(p[0][:2]), np.diff(p[1][:2]))[0]
                for p in (lattices(descs) if overlaps else parts))
    assert g.min_distance() == pytest.approx(least, rel=1e-12)
    g.close()
