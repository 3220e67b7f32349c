"""The library's host code on a fake CUDA runtime of two devices (fake_cuda.cpp).  A
phi-set destroyed while another device is current (a garbage collector does that)
returns its memory to its own device, behind that device's work.  What the library's
memory pool keeps is given back before another allocation is refused."""
import glob
import os
import re
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(ROOT, "paper_2310_07551_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc, tmp = os.path.join(CUDA, "bin", "nvcc"), tmp_path_factory.mktemp("fake")
    if shutil.which("g++") is None or not os.path.exists(nvcc):
        pytest.skip("no compilers")
    objs = [str(tmp / (n + ".o")) for n in ("api", "step64")]
    for o in objs:
        src = os.path.join(CSRC, os.path.basename(o)[:-1] + "cu")
        subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "--expt-relaxed-constexpr", "-c", src,
                        "-o", o], check=True)
    prog = str(tmp / "prog")
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(CUDA, "include"), "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    os.path.join(HERE, "fake_cuda.cpp"), *objs, "-o", prog, "-Wl,--unresolved-symbols=ignore-all"], check=True)
    return prog


@pytest.mark.parametrize("what", ["destroy", "scarce"])
def test_on_a_fake_runtime(program, what):
    r = subprocess.run([program, what], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


def test_every_allocation_empties_the_pool_first():
    """cudaMalloc is called by the one function that does"""
    calls = [(os.path.basename(f), line.strip()) for f in sorted(glob.glob(os.path.join(CSRC, "*")))
             for line in open(f) if re.search(r"\bcudaMalloc\(", line)]
    assert calls and {f for f, _ in calls} == {"api.cu"} and len(calls) == 2, calls
