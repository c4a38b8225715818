"""Memory order between the lanes of the hard-sphere cells, on the CPU: their
device code on the fibers of warp_lanes.h under ThreadSanitizer, where only
__syncwarp orders memory.
"""
import os
import re

import pytest

import lanes

# k, eta, cells per side, ell, n_m, rel, shortest
CASES = {
    "small_cells": "8 0.40 4 2.0 4 1 0",
    "unscreened_frames": "8 0.40 4 8.0 3 0 0",
    "images_of_a_two_cell_box": "8 0.40 2 8.0 3 0 1",
    "bins_and_dropped_lists": "16 0.40 4 4.0 6 1 1",
    "long_rattles": "16 0.40 8 30.0 3 1 0",
}


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("lanes")
    # the device code, with the dynamic shared memory as an array and no clock
    with open(os.path.join(lanes.CSRC, "ecmc3.cu")) as f:
        text = f.read().split("// ---- host side")[0]
    clock = 'asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));'
    smem = "  extern __shared__ __align__(16) unsigned char smem[];\n"
    assert text.count(clock) == 1 and smem in text
    text = text.replace(clock, "t = 0;").replace(smem, "").replace(
        "namespace ecmc3 {\n", "namespace ecmc3 {\nextern unsigned char smem[232448];\n", 1)
    (d / "spheres_device.h").write_text(text)
    return lanes.build(d, "sphere_lanes.cpp",
                       {"spheres": ['-DSPHERES="%s"' % (d / "spheres_device.h")]})["spheres"]


@pytest.mark.parametrize("case", sorted(CASES))
def test_lanes_order_their_memory(program, case):
    up, down = (lanes.run(program, CASES[case] + d) for d in (" 0", " 1"))
    assert up == down
    n = {k: int(v) for k, v in re.findall(r"(\w+) (\d+) ", up[0])}
    assert n["lifts"] > 0 and n["frozen"] > 0 and n["replayed"] > 0
