"""A phi-set destroyed while another device is current (a garbage collector does that)
returns its memory to its own device, behind that device's work: the library's host code
on a fake CUDA runtime of two devices."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


@pytest.mark.skipif(shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "bin", "nvcc")), reason="no compilers")
def test_destroy_frees_on_the_set_s_own_device(tmp_path):
    pkg = os.path.join(ROOT, "paper_2310_07551_gb300")
    obj, prog = str(tmp_path / "api.o"), str(tmp_path / "prog")
    subprocess.run([os.path.join(CUDA, "bin", "nvcc"), "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17",
                    "--expt-relaxed-constexpr", "-c", os.path.join(pkg, "csrc", "api.cu"), "-o", obj], check=True)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(CUDA, "include"), "-I", os.path.join(pkg, "csrc"),
                    "-I", os.path.join(ROOT, "include"), os.path.join(HERE, "fake_cuda.cpp"), obj, "-o", prog,
                    "-Wl,--unresolved-symbols=ignore-all"], check=True)
    r = subprocess.run([prog], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
