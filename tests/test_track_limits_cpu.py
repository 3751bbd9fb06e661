"""Tracking windows and bursts past the kernels' index ranges are refused before anything is launched (the plan is
filled in by hand: a real one needs a GPU)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <cstdio>
#include <cstdlib>
#include "sm_plan.h"
int main(int argc, char** argv) {
    sm_plan pl;
    pl.dev.W = pl.dev.H = 65536;
    alignas(16) static char mem[16];
    const int rc = sm_stage_track(&pl, mem, SM_F32, atoi(argv[1]), 0, atoi(argv[2]), atoi(argv[3]), (float*)mem,
                                  (double*)mem, (int*)mem, nullptr);
    printf("%d %s\n", rc, sm_last_error());
}
"""


@pytest.fixture(scope="module")
def track(tmp_path_factory):
    from paper_1701_00581_gb300 import build
    lib = build.build()
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("track")
    (d / "track.cpp").write_text(SRC)
    subprocess.run([cxx, "-std=c++17", "-I", build.INCLUDE, "-I", build.CSRC, "-I",
                    os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include"), str(d / "track.cpp"),
                    lib, "-Wl,-rpath," + os.path.dirname(lib), "-o", str(d / "track")], check=True)
    return lambda *a: subprocess.run([str(d / "track"), *map(str, a)], capture_output=True, text=True, check=True).stdout


# one past G + S = 29056; the first G whose G * G samples overflow an int; the largest that fits the frame; F past a
# grid's second dimension
@pytest.mark.parametrize("F,G,S", [(1, 29057, 0), (1, 29040, 17), (2, 46341, 16), (1, 65536, 0), (65536, 64, 4)])
def test_refused(track, F, G, S):
    from paper_1701_00581_gb300 import _lib
    rc, _, msg = track(F, G, S).partition(" ")
    assert int(rc) == _lib.SM_EINVAL and "29056" in msg
