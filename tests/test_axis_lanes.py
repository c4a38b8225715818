"""Memory order between the lanes of the axis-chain kernel, on the CPU.

csrc/ecmc_axis.cuh runs on 32 fibers under ThreadSanitizer (warp_lanes.h): votes
and shuffles exchange values but order no memory, __syncwarp does.  A word that
one lane writes and another reads or writes without a __syncwarp between them
is reported as a data race.  Results must not depend on the order in which the
lanes run, nor on the number of lanes per cell.
"""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "include/cuda_runtime.h")):
    pytest.skip("needs g++ and the CUDA headers", allow_module_level=True)

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
    d = tmp_path_factory.mktemp("lanes")
    probe = d / "probe"
    (d / "probe.cpp").write_text("int main() { return 0; }\n")
    if subprocess.run(["g++", "-fsanitize=thread", str(d / "probe.cpp"), "-o", str(probe)],
                      capture_output=True).returncode or \
            subprocess.run([str(probe)], capture_output=True).returncode:
        pytest.skip("ThreadSanitizer does not run here")
    flags = ["-std=c++20", "-O1", "-g", "-Wno-unknown-pragmas"]
    lanes_o = str(d / "warp_lanes.o")
    subprocess.run(["g++", *flags, "-fno-tree-loop-distribute-patterns", "-c",
                    os.path.join(HERE, "warp_lanes.cpp"), "-o", lanes_o], check=True)
    jobs, out = [], {}
    for n in LANES:
        out[n] = str(d / ("axis_lanes%d" % n))
        jobs.append(subprocess.Popen(
            ["g++", *flags, "-fsanitize=thread", "-DLANES=%d" % n,
             "-I", os.path.join(CUDA, "include"), "-I", os.path.join(ROOT, "include"),
             "-I", os.path.join(ROOT, "paper_1409_6948_gb300", "csrc"),
             os.path.join(HERE, "axis_lanes.cpp"), lanes_o, "-o", out[n]]))
    assert [j.wait() for j in jobs] == [0] * len(jobs)
    return out


def run(program, case, downwards):
    r = subprocess.run([program, *CASES[case].split(), str(downwards)], capture_output=True,
                       text=True, timeout=300, env={**os.environ, "TSAN_OPTIONS": "atexit_sleep_ms=0"})
    races = r.stderr.count("WARNING: ThreadSanitizer")
    assert races == 0, "%d data races\n%s" % (races, r.stderr[:4000])
    assert r.returncode == 0, r.stdout + r.stderr[:4000]
    return r.stdout.splitlines()


@pytest.mark.parametrize("case", sorted(CASES))
def test_lanes_order_their_memory(programs, case):
    first = None
    for n in LANES:
        up, down = run(programs[n], case, 0), run(programs[n], case, 1)
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
