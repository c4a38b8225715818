"""The three-dimensional overlap check on fixed-point positions, against the
oracle's grid search, bit for bit: cells of every occupation class, the box
sizes where the FP64 scan takes over, exact ties and planted near-ties.
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


def check(N, L, cells, xyz):
    g = P.Ecmc3(N, L, 1.0, cells, 1.0, 3)
    g.set_positions(xyz)
    x, y, z = (np.ascontiguousarray(xyz[a::3]) for a in range(3))
    rc = min(2.0, L / cells)
    assert g.min_distance() == math.sqrt(oracle.min_dist2_3(L, x, y, z, rc))
    g.close()


@pytest.mark.parametrize("N,eta,cells", [
    (4096, 0.45, 8),     # about 8 members per cell
    (4096, 0.45, 6),     # 19: lanes in groups of 16 and 32
    (4096, 0.40, 4),     # 64: several rounds of lanes
    (4096, 0.45, 14),    # cells narrower than 2 sigma bound the search
    (1000, 0.30, 2),     # two cells per side: the FP64 scan
    (216, 0.30, 4),      # a box below 8 sigma: the FP64 scan
])
@pytest.mark.parametrize("jitter", [0.0, 1.0])
def test_lattices_bitwise(N, eta, cells, jitter):
    # jitter 0: every nearest distance of the cubic lattice ties
    L = W.box_side3(N, eta)
    a = L / round(N ** (1 / 3))
    rng = np.random.default_rng(N + cells)
    u = (rng.random((N, 3)) - 0.5) * jitter * 0.98 * (a - 1.0)
    xyz = (np.stack(W.cubic_lattice(N, L), 1) + u) % L
    check(N, L, cells, xyz.ravel())


@pytest.mark.parametrize("seed", range(4))
def test_planted_near_ties(seed):
    # pairs at 1.5 sigma but for a few ulps, across the boundary too: only FP64
    # can order them
    k, a = 8, 3.0
    N, L = k ** 3, k * a
    rng = np.random.default_rng(seed)
    xyz = np.stack(W.cubic_lattice(N, L), 1)
    for i, axis in ((0, 0), (70, 1), (200, 2), (N - 1, 0)):
        step = 1 if axis == 0 else (k if axis == 1 else k * k)
        j = (i + step) % N
        xyz[j] = xyz[i]
        xyz[j, axis] = (xyz[i, axis] + 1.5 + float(rng.integers(-3, 4)) * 2.0 ** -50) % L
    check(N, L, 8, xyz.ravel())
