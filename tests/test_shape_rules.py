"""The host rules that choose a sweep kernel, without a GPU: a small program
linked against the library prints what the rules say for given sizes."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
OPTIN = 227 << 10

SOURCE = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "spvar_internal.h"
using namespace spvar;
int main(int argc, char **argv)
{
    auto arg = [&](int i) { return i < argc ? std::atoi(argv[i]) : 0; };
    if (!std::strcmp(argv[1], "request")) {
        // block, n, quads, degree: taken as a request, shared memory of the launch, second table
        const QuadLayout l = pm1q_layout(arg(2), arg(3), arg(4), arg(5));
        std::printf("%d %zu %d\n", (int)pm1q_request_ok(arg(2), arg(3), arg(4), arg(5), kSmemOptin), l.bytes + l.stat,
                    (int)l.tabs);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    from paper_1706_07826_gb300 import build as B
    lib = B.build()
    d = tmp_path_factory.mktemp("rules")
    (d / "rules.cpp").write_text(SOURCE)
    subprocess.run([nvcc, "-std=c++17", "-I", B.CSRC, "-I", B.INCLUDE, str(d / "rules.cpp"), lib, "-cudart", "shared",
                    "-Xlinker", "-rpath," + os.path.dirname(lib), "-o", str(d / "rules")], check=True)
    return lambda *a: subprocess.run([str(d / "rules")] + [str(x) for x in a], check=True, capture_output=True,
                                     text=True).stdout.split()


@pytest.mark.parametrize("maxd", [6, 8])
def test_requested_quads_are_taken_where_the_launch_fits(rules, maxd):
    """One quad per item: every size up to 28585 spins, as with one quad per
    word, and none whose launch does not fit a block's shared memory."""
    for n in (27000, 28200, 28275, 28276, 28400, 28585, 28787, 28788, 28800, 29055):
        ok, smem, tabs = rules("request", 256, n, 1, maxd)
        assert int(ok) == (int(smem) <= OPTIN)
        if n <= 28585:
            assert int(ok) == 1
        if n < 28200:
            assert int(tabs) == (maxd == 6)
    assert rules("request", 256, 28800, 1, maxd)[0] == "0"
