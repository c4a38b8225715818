"""The end-of-sweep sums over two and over more than 32 chunks of 2048 cells:
counters and pressure against the oracle's, as in test_gpu_parity."""
import pytest

from test_gpu_parity import run_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,eta,cells,ell,nm", [
    (90000, 0.30, 258, 1.0, 1),   # 66,564 cells: 33 chunks
    (10000, 0.30, 64, 1.0, 2),    # two chunks
])
def test_totals_match_oracle(N, eta, cells, ell, nm):
    run_pair(N, eta, cells, cells, ell, nm, 23, 2)
