"""Memory order between the threads of the stripes' sorted-frame kernel, on the
CPU: its device code on the fibers of warp_lanes.h under ThreadSanitizer, where
only __syncwarp and __syncthreads order memory.
"""
import os
import re

import pytest

import lanes

# columns, rows, L, stripes, ell, n_m, reject, list mode
CASES = {
    "rejected": "21 26 25.4 4 2.0 30 1 0",
    "rejected_shuffled": "21 26 25.4 4 2.0 30 1 1",
    "reflected": "21 26 25.4 4 6.0 4 0 0",
    "reflected_round_the_box": "21 26 25.4 2 60.0 2 0 1",
}


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("lanes")
    # the device code, with the dynamic shared memory as an array
    with open(os.path.join(lanes.CSRC, "ecmc_stripes.cu")) as f:
        text = f.read().split("// ---- host side")[0]
    smem = "  extern __shared__ __align__(16) unsigned char ssm[];\n"
    assert text.count(smem) == 1
    text = text.replace(smem, "").replace(
        "namespace ecmcs {\n", "namespace ecmcs {\nextern unsigned char ssm[232448];\n", 1)
    (d / "stripes_device.h").write_text(text)
    return lanes.build(d, "stripe_lanes.cpp",
                       {"stripes": ['-DSTRIPES="%s"' % (d / "stripes_device.h")]})["stripes"]


@pytest.mark.parametrize("case", sorted(CASES))
def test_threads_order_their_memory(program, case):
    up, down = (lanes.run(program, CASES[case] + d) for d in (" 0", " 1"))
    assert up == down
    n_rej = sum(int(m) for m in re.findall(r"rejected (\d+)", "\n".join(up)))
    n_ch = sum(int(m) for m in re.findall(r"chains (\d+)", "\n".join(up)))
    assert (0 < n_rej < n_ch) if case.startswith("rejected") else n_rej == 0
