"""The host planner's tables (plan_host.cpp), against the definition of a used pair, and the time they take."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def plan_host(tmp_path_factory):
    from paper_1701_00581_gb300 import build
    build.build()
    nvcc = build._nvcc()
    lib = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "lib64")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(lib, "libcudart.so")):
        pytest.skip("no C++ compiler or shared CUDA runtime")
    exe = str(tmp_path_factory.mktemp("plan") / "plan_host")
    objs = [os.path.join(build.BUILD, os.path.splitext(f)[0] + ".o") for f in build.CU_SOURCES + build.CPP_SOURCES]
    subprocess.run([nvcc, "-O2", "-std=c++17", "-cudart", "shared", "-I", build.INCLUDE, "-I", build.CSRC, "-o", exe,
                    os.path.join(HERE, "plan_host.cpp"), *objs, "-Xlinker", "-rpath," + lib], check=True)

    def run(*args):
        r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stdout
        return r.stdout
    return run


# both parities of the radius and the cutoff, one offset, radii up to the cutoff, every phasor size
@pytest.mark.parametrize("N,R,fc,prec", [(64, 1, 0.2885, 0), (64, 8, 0.2885, 0), (64, 7, 0.25, 2), (64, 18, 0.2885, 1),
                                         (64, 3, 0.05, 0), (128, 16, 0.2885, 0), (128, 33, 0.27, 2), (256, 5, 0.2, 1),
                                         (256, 24, 0.2885, 0)])
def test_tables(plan_host, N, R, fc, prec):
    assert plan_host(N, R, fc, prec).startswith("0 wrong")


@pytest.mark.parametrize("N,R", [(128, 16), (256, 24)])
def test_time(plan_host, N, R):
    """All of a plan's tables in less time than testing every slot of every tile once, on the same machine (the best
    of three, since others may be running)."""
    ratio = []
    for _ in range(3):
        plan, slots = map(float, re.search(r"plan ([\d.]+) ms, slots ([\d.]+) ms", plan_host(N, R, 0.2885, 0)).groups())
        ratio.append(plan / slots)
    assert min(ratio) < 1.0, ratio
