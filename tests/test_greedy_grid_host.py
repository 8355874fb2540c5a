"""The greedy pass's launch size (paper_2609_33224_gb300/csrc/greedy_grid.h): its blocks wait on one another,
so a launch may hold no more of them than fit on the device at once, on a whole GPU or on a part of one."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_33224_gb300", "csrc")

HARNESS = r"""
#include <cstdio>
#include "greedy_grid.h"
int main() {
  unsigned R, lag, resident;
  while (std::scanf("%u %u %u", &R, &lag, &resident) == 3) {
    const psgrid::PipeGrid g = psgrid::pipe_grid(R, lag, resident);
    std::printf("%u %u %u\n", g.insert, g.probe, g.blocks());
  }
}
"""


@pytest.fixture(scope="module")
def grid(tmp_path_factory):
    d = tmp_path_factory.mktemp("grid")
    src, exe = d / "g.cpp", d / "g"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)

    def run(cases):
        text = "".join("%d %d %d\n" % c for c in cases)
        out = subprocess.run([str(exe)], input=text, capture_output=True, check=True, text=True).stdout
        return [tuple(int(x) for x in line.split()) for line in out.splitlines()]
    return run


def test_launches_fit_the_device(grid):
    cases = [(R, 33, sms) for R in (1, 2, 5, 8, 33, 34, 40, 63, 64, 65, 500, 131072) for sms in range(1, 200)]
    for (R, lag, sms), (insert, probe, blocks) in zip(cases, grid(cases)):
        assert blocks == 1 + insert + probe <= max(sms, 6), (R, sms)
        assert 1 <= probe <= min(R, 64) and insert % 4 == 0 and insert <= 64, (R, sms)
        assert (insert >= 4) == (R > lag), (R, sms)
        full = (64 if R > lag else 0) + min(R, 64)
        assert insert + probe == full if 1 + full <= sms else insert + probe > min(full, max(sms, 6) - 1) - 4, (R, sms)


def test_the_whole_device_takes_the_full_launch(grid):
    assert grid([(16384, 33, 152), (40, 33, 152), (33, 33, 152), (1, 33, 152)]) == [
        (64, 64, 129), (64, 40, 105), (0, 33, 34), (0, 1, 2)]
