"""A batch's device queue (batch_host.cpp): every transform and every bispectrum task once, transforms before the tasks
that read them, and sm_batch_info's count of what the queue covers."""
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def batch_host(tmp_path_factory):
    from paper_1701_00581_gb300 import build
    build.build()
    nvcc = build._nvcc()
    lib = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "lib64")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(lib, "libcudart.so")):
        pytest.skip("no C++ compiler or shared CUDA runtime")
    exe = str(tmp_path_factory.mktemp("batch") / "batch_host")
    objs = [os.path.join(build.BUILD, os.path.splitext(f)[0] + ".o") for f in build.CU_SOURCES + build.CPP_SOURCES
            if f != "sm_batch.cpp"]
    subprocess.run([nvcc, "-O2", "-std=c++17", "-cudart", "shared", "-I", build.INCLUDE, "-I", build.CSRC, "-o", exe,
                    os.path.join(HERE, "batch_host.cpp"), *objs, "-Xlinker", "-rpath," + lib], check=True)
    return exe


@pytest.mark.parametrize("launch", [1, 2])                 # SM_BATCH_FUSED, SM_BATCH_TILES
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("lookahead", [1, 3, 1000])        # past the batch's last subfield too
def test_queue(batch_host, launch, order, lookahead):
    r = subprocess.run([batch_host, str(launch), str(order), str(lookahead)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.startswith("0 wrong"), r.stdout


def test_lookahead_by_default(batch_host):
    """Left to itself a fused queue's transforms run ahead by twice the subfields whose items the CTAs hold at once, so
    that none of those waits for another; a given lookahead stays as it is."""
    def run(lookahead):
        out = subprocess.run([batch_host, "1", "2", str(lookahead)], capture_output=True, text=True, check=True).stdout
        return [int(v) for v in re.search(r"lookahead (\d+), in flight (\d+) of (\d+)", out).groups()]
    ahead, flight, items = run(0)
    assert flight == 4 * 152 and ahead * items >= 2 * flight > (ahead - 1) * items
    assert run(3)[0] == 3
