"""Hard spheres: the members' candidate lists and the frame's FP32 screen at
the edges of their ranges, against the oracle.

Cells are compared through binning, chain records, positions and counters.
Cases: one sphere and a handful, two cells per side (several images, no
screen), frames with and without bins across the axis, so many chains per
cell that the lists fill their room and are dropped and found again, dense
and dilute systems.
"""
import pytest

from test_gpu3 import run_pair3

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("persistent", [1, 0])
@pytest.mark.parametrize("N,eta,cells,ell,nm,sweeps", [
    (1, 0.05, 2, 3.0, 2, 6),
    (8, 0.10, 2, 4.0, 6, 6),
    (512, 0.30, 2, 1.5, 40, 4),
    (1728, 0.50, 6, 2.0, 20, 4),      # no bins, lists dropped
    (2744, 0.45, 4, 2.0, 60, 3),      # bins, lists dropped
    (4096, 0.02, 8, 30.0, 4, 3),
])
def test_lists_match_oracle(N, eta, cells, ell, nm, sweeps, persistent):
    run_pair3(N, eta, cells, ell, nm, 17, sweeps, persistent)
