"""Which copies one kernel may make (csrc/copy_route.cuh), compiled for the
host: only of arrays in the context's own device's memory, while that device is
current.  Two devices, whatever is current, without a GPU."""
import itertools
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2606_03770_gb300", "csrc")
CASES = list(itertools.product((0, 1), (0, 1), (0, 1), (0, 1)))    # device memory, its owner, the context's device, current


@pytest.fixture(scope="module")
def route(tmp_path_factory):
    d = tmp_path_factory.mktemp("route")
    (d / "route.cpp").write_text(
        '#include "copy_route.cuh"\n#include <cstdio>\n#include <cstdlib>\n'
        'int main(int, char **a) { std::printf("%d", e2::copied_by_kernel(std::atoi(a[1]), std::atoi(a[2]), '
        'std::atoi(a[3]), std::atoi(a[4]))); }\n')
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "route.cpp"), "-o", str(d / "route")], check=True)
    return lambda *x: subprocess.run([str(d / "route"), *map(str, x)], check=True, capture_output=True, text=True).stdout


@pytest.mark.parametrize("device_memory,owner,context,current", CASES)
def test_copied_by_kernel(route, device_memory, owner, context, current):
    # (a launch on the context's stream needs its device to be current, and no peer access is asked for)
    want = device_memory == 1 and owner == context == current
    assert route(device_memory, owner, context, current) == str(int(want))
