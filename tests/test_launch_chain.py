"""What the ring leaves for the FP64 analysis and its finish is cleared when one
of the two is not launched (fakes of the launches that return an error code)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1009_3308_gb300", "csrc")

MAIN = r"""
#include "chain.h"
#include <cstdio>
#include <cstdlib>
int main(int, char** v) {
    const int r1 = std::atoi(v[1]), r2 = std::atoi(v[2]);
    int emax = 5, calls = 0;   // raised by the ring
    const int rc = sph::chain_or_reset([&] { ++calls; return r1; },
                                       [&] { ++calls; if (!r2) emax = 0; return r2; }, [&] { emax = 0; });
    std::printf("%d %d %d\n", rc, calls, emax);
}
"""


@pytest.mark.parametrize("r1,r2,want", [(0, 0, "0 2 0"), (-3, 0, "-3 1 0"), (0, -4, "-4 2 0")])
def test_exponents_do_not_outlive_a_failed_launch(tmp_path, r1, r2, want):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe), str(r1), str(r2)], check=True, capture_output=True, text=True).stdout
    assert out.strip() == want


def test_the_fp64_analysis_uses_it():
    src = open(os.path.join(CSRC, "plan.cu")).read()
    body = src[src.index("static int analysis64("):]
    body = body[:body.index("\n}\n")]
    assert "chain_or_reset(" in body and "dig_clear_exponents" in body
