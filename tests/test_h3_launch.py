"""Launch shape of the FP16 x3 detection kernel (detect_h3.cuh), from its compile-time constants (no GPU).

A CTA of this kernel holds all of its SM's TMEM while it waits for the other CTAs of its cluster, so two
must never share an SM: the second would wait in its TMEM allocation, and two clusters placed on two SMs
in opposite order would wait for each other."""
import os
import re
import subprocess

import pytest

from paper_2201_05024_gb300 import build

SM_SHARED, CTA_RESERVED = 228 * 1024, 1024  # shared memory of an SM; what the system keeps per CTA

SOURCE = r"""
#include <cstdio>
#include "detect_h3.cuh"
using namespace apsm;
template <int M, int KB> void show() { std::printf("%d %d %d %d\n", M, KB, H3Smem<M, KB>::kBytes, H3Smem<M, KB>::kLaunch); }
template <int M> void row() { show<M, 2>(); show<M, 4>(); show<M, 6>(); show<M, 8>(); show<M, 12>(); show<M, 16>(); }
int main() { row<16>(); row<32>(); row<64>(); }
"""


@pytest.fixture(scope="module")
def footprints(tmp_path_factory):
    d = tmp_path_factory.mktemp("h3")
    (d / "show.cu").write_text(SOURCE)
    exe = str(d / "show")
    r = subprocess.run([build._nvcc(), *build.ARCH, "-O0", "-std=c++17", "--expt-relaxed-constexpr",
                        "-I" + os.path.join(build.ROOT, "include"), "-I" + build.CSRC, str(d / "show.cu"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout
    return [tuple(map(int, line.split())) for line in out.splitlines()]


def test_no_two_ctas_of_any_instantiations_fit_an_sm(footprints):
    assert len(footprints) == 18
    smallest = min(launch for *_, launch in footprints)
    assert 2 * (smallest + CTA_RESERVED) > SM_SHARED
    for _, _, used, launch in footprints:
        assert used <= launch <= SM_SHARED - CTA_RESERVED


def test_launch_and_occupancy_query_ask_for_it():
    """The figure above is what the launch configuration (which the cluster query reads too) carries."""
    src = open(os.path.join(build.CSRC, "detect_h3.cuh")).read()
    asked = re.findall(r"(?:dynamicSmemBytes = |MaxDynamicSharedMemorySize, )(L::\w+)", src)
    assert asked == ["L::kLaunch", "L::kLaunch"]
