"""Builds and runs the programs that put device code on the fibers of
warp_lanes.h under ThreadSanitizer."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_1409_6948_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")
FLAGS = ["-std=c++20", "-O1", "-g", "-Wno-unknown-pragmas"]


def build(d, source, variants):
    """Compile tests/<source> once per entry {name: flags} of variants into d."""
    if shutil.which("g++") is None or \
            not os.path.exists(os.path.join(CUDA, "include/cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    probe = d / "probe"
    (d / "probe.cpp").write_text("int main() { return 0; }\n")
    if subprocess.run(["g++", "-fsanitize=thread", str(d / "probe.cpp"), "-o", str(probe)],
                      capture_output=True).returncode or \
            subprocess.run([str(probe)], capture_output=True).returncode:
        pytest.skip("ThreadSanitizer does not run here")
    lanes_o = str(d / "warp_lanes.o")
    subprocess.run(["g++", *FLAGS, "-fno-tree-loop-distribute-patterns", "-c",
                    os.path.join(HERE, "warp_lanes.cpp"), "-o", lanes_o], check=True)
    out = {name: str(d / ("lanes_%s" % name)) for name in variants}
    jobs = [subprocess.Popen(
        ["g++", *FLAGS, "-fsanitize=thread", *flags, "-I", os.path.join(CUDA, "include"),
         "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-I", HERE,
         os.path.join(HERE, source), lanes_o, "-o", out[name]])
        for name, flags in variants.items()]
    assert [j.wait() for j in jobs] == [0] * len(jobs)
    return out


def run(program, args):
    """The program's output lines; fails on a data race."""
    r = subprocess.run([program, *args.split()], capture_output=True, text=True, timeout=300,
                       env={**os.environ, "TSAN_OPTIONS": "atexit_sleep_ms=0"})
    races = r.stderr.count("WARNING: ThreadSanitizer")
    assert races == 0, "%d data races\n%s" % (races, r.stderr[:4000])
    assert r.returncode == 0, r.stdout + r.stderr[:4000]
    return r.stdout.splitlines()
