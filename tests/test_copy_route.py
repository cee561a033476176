"""Which copies one kernel may make (csrc/copy_route.cuh), compiled for the
host: only of arrays in the context's own device's memory, while that device is
current (two devices, whatever is current, without a GPU), and of outputs that
share no byte."""
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
        'int main(int n, char **a) { int x[4]; for (int i = 0; i < 4; ++i) x[i] = std::atoi(a[2 + i]);\n'
        '  static unsigned char m[64];\n'
        '  std::printf("%d", a[1][0] == \'k\' ? e2::copied_by_kernel(x[0], x[1], x[2], x[3])\n'
        '                                   : e2::overlap(m + x[0], x[1], m + x[2], x[3])); }\n')
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(d / "route.cpp"), "-o", str(d / "route")], check=True)
    return lambda *x: subprocess.run([str(d / "route"), *map(str, x)], check=True, capture_output=True, text=True).stdout


@pytest.mark.parametrize("device_memory,owner,context,current", CASES)
def test_copied_by_kernel(route, device_memory, owner, context, current):
    # (a launch on the context's stream needs its device to be current, and no peer access is asked for)
    want = device_memory == 1 and owner == context == current
    assert route("k", device_memory, owner, context, current) == str(int(want))


@pytest.mark.parametrize("a,na,b,nb", [(0, 8, 8, 8), (8, 8, 0, 8), (0, 8, 7, 8), (7, 8, 0, 8), (4, 4, 0, 32), (0, 32, 4, 1),
                                       (3, 5, 3, 5), (0, 1, 2, 1)])
def test_overlap(route, a, na, b, nb):
    assert route("o", a, na, b, nb) == str(int(bool(set(range(a, a + na)) & set(range(b, b + nb)))))
