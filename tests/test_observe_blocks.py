"""The observables' launch on the host: whatever the number of SMs, no thread
counts more arms of one state than its 16-bit lanes hold (CPU only: a host
program around the launch's rule)."""
import os
import subprocess

import pytest

from paper_2505_05919_gb300 import build as libbuild

PROGRAM = """
#include <cstdio>
#include <cstdlib>
#include "cvf_observe.cuh"
int main(int argc, char** argv) {
  for (int i = 1; i + 2 < argc; i += 3)
    std::printf("%d\\n", cvf::observe_blocks(std::atoll(argv[i]), std::atoi(argv[i + 1]), std::atoi(argv[i + 2])));
}
"""


@pytest.fixture(scope="module")
def blocks(tmp_path_factory):
    d = tmp_path_factory.mktemp("observe")
    src, exe = str(d / "blocks.cu"), str(d / "blocks")
    open(src, "w").write(PROGRAM)
    subprocess.run([libbuild.nvcc()] + libbuild.ARCH + ["-std=c++17", "-I" + libbuild.INCLUDE,
                   "-I" + libbuild.CSRC, src, "-o", exe], check=True, capture_output=True)

    def run(cases):
        out = subprocess.run([exe] + [str(x) for c in cases for x in c], check=True,
                             capture_output=True, text=True, env=dict(os.environ)).stdout
        return [int(x) for x in out.split()]
    return run


def test_no_lane_overflows_on_any_number_of_sms(blocks):
    cases = [(L * L, sms, 4) for L in (2, 32, 1024, 4096, 16384, 65534) for sms in (1, 16, 64, 127, 152)]
    cases += [(L ** 3, sms, 6) for L in (2, 3, 51, 260, 1021, 1024) for sms in (1, 16, 64, 127, 152)]
    for (N, sms, arms), b in zip(cases, blocks(cases)):
        loads = (N + 3) // 4
        used = min(b, (loads + 255) // 256)              # as the kernel does
        a_thread = (loads + 256 * used - 1) // (256 * used)
        assert b >= 1 and 4 * arms * a_thread <= 65535, (N, sms, arms, b)


def test_the_launch_on_152_sms(blocks):
    # unchanged: two loads a thread for small lattices, 8 blocks an SM beyond
    cases = [(32 * 32, 152, 4), (1024 * 1024, 152, 4), (65534 ** 2, 152, 4), (1024 ** 3, 152, 6)]
    assert blocks(cases) == [1, 512, 1216, 1216]
