"""Isotropic chains with every number of lanes per cell against the oracle:
one lane computes both components of a vector, two or more share them; the
exact wall distances are skipped where their FP32 bounds leave no doubt.

Positions, records and counters as in test_gpu_parity.  Cases: cells little
wider than sigma and dilute (nearly every leg ends at a wall), dense and
rectangular cells, long chains, several groups of lanes at a tie of many
candidates (the square-lattice start).
"""
import pytest

from test_gpu_parity import run_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [1, 0])
@pytest.mark.parametrize("tpc", [1, 2, 4, 8, 16, 32])
@pytest.mark.parametrize("N,eta,cx,cy,ell,nm,sweeps", [
    (64, 0.05, 24, 24, 9.0, 2, 4),
    (1024, 0.71, 8, 4, 3.0, 2, 3),
    (576, 0.60, 12, 12, 0.7, 3, 4),
])
def test_lanes_match_oracle(N, eta, cx, cy, ell, nm, sweeps, tpc, prec):
    run_pair(N, eta, cx, cy, ell, nm, 19, sweeps, tpc=tpc, prec=prec, dir_mode=2)
