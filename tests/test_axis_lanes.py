"""Memory order between the lanes of the axis-chain kernel, on the CPU.

csrc/ecmc_axis.cuh runs on 32 fibers under ThreadSanitizer (warp_lanes.h): votes
and shuffles exchange values but order no memory, __syncwarp does.  A word that
one lane writes and another reads or writes without a __syncwarp between them
is reported as a data race.  Results must not depend on the order in which the
lanes run, nor on the number of lanes per cell.
"""
import re

import pytest

import lanes

LANES = (2, 4, 8, 32)
# k, eta, cells per side, ell, n_m, boundary, list mode, start
CASES = {
    "turn_backs": "32 0.70 8 2.0 6 0 0 0",
    "cycles": "32 0.70 8 30.0 3 0 0 0",
    "more_chains_than_draws": "32 0.70 8 0.5 40 0 0 0",
    "shuffled_list": "32 0.70 8 2.0 6 0 1 0",
    "rejected": "32 0.70 8 0.05 40 1 0 0",
    "rejected_shuffled": "32 0.70 8 0.05 40 1 1 0",
    "whole_frame_search": "32 0.74 8 3.0 3 0 0 1",
    "whole_frame_search_rejected": "32 0.74 8 0.5 20 1 0 1",
}


@pytest.fixture(scope="module")
def programs(tmp_path_factory):
    return lanes.build(tmp_path_factory.mktemp("lanes"), "axis_lanes.cpp",
                       {n: ["-DLANES=%d" % n] for n in LANES})


@pytest.mark.parametrize("case", sorted(CASES))
def test_lanes_order_their_memory(programs, case):
    first = None
    for n in LANES:
        up, down = (lanes.run(programs[n], CASES[case] + " 1" + d)[:-1] for d in (" 0", " 1"))
        assert up == down
        assert len(up) == min(16, 32 // n)
        # how much of a chain is replayed depends on the lanes, what it does not
        cells = [re.sub(r"replayed \d+ |sum_b \S+ ", "", line) for line in up]
        if first is None:
            first = cells
        assert cells == first[:len(cells)]
    assert any(" irregular 1:" in c for c in first) == case.startswith("whole_frame")
    # rejected some, accepted some
    n_rej = sum(int(re.search(r"rejected (\d+)", c).group(1)) for c in first)
    n_ch = sum(int(re.search(r"chains (\d+)", c).group(1)) for c in first)
    assert (0 < n_rej < n_ch) if "rejected" in case else n_rej == 0


@pytest.mark.parametrize("n", LANES)
def test_fp64_candidates_are_chosen_in_fp64(programs, n):
    # the same candidates either way; FP32 leaves next to nothing to FP64 here,
    # and the FP64 setting compares every object of a window's strips
    case = CASES["turn_backs"]
    fp32, fp64 = (lanes.run(programs[n], case + p) for p in (" 1 0", " 0 0"))
    assert fp32[:-1] == fp64[:-1]
    counts = [[int(v) for v in re.findall(r"\d+", x[-1].replace("fp64", ""))]
              for x in (fp32, fp64)]
    members = counts[0][0]
    assert counts[0][1] < members < 3 * members <= counts[1][1]
