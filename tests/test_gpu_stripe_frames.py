"""The frames of the striped decomposition at the edges of their construction
(sorted-frame kernel, include/ecmc_stripes.h) against the oracle.

Positions, stripes, chain records and counters must match exactly: boxes so
small that fewer warps than a block's take part and a strip is one bucket,
stripes of width sigma up to rounding (disks two stripes away are looked at),
two stripes (images at +-L count), runs of more than 256 ids, a long box of
few wide stripes.
"""
import math

import pytest

from test_gpu_stripes import REFLECT, REJECT, run_pair

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k,L,S,ell,nm,sweeps,boundary", [
    (1, 2.5, 2, 3.0, 2, 6, REJECT),
    (2, 2.2, 2, 1.5, 3, 6, REFLECT),
    (3, 4.5, 4, 2.0, 2, 6, REJECT),
    (15, 16.0 * (1.0 + 4e-13), 16, 2.0, 3, 6, REFLECT),
    (16, 17.5, 2, 6.0, 3, 6, REJECT),
    (17, 20.0, 4, 9.0, 2, 6, REFLECT),
    (300, 322.0, 64, 2.0, 2, 2, REJECT),
])
def test_frames_match_oracle(k, L, S, ell, nm, sweeps, boundary):
    run_pair(k * k, k * k * math.pi / (4.0 * L * L), S, ell, nm, 31, sweeps, boundary)
