"""CPU test of the library's host logic around the GPU: its own objects linked with a fake CUDA runtime
(tests/fake_cuda_check.cpp) that keeps device memory on the host and records every allocation,
clear and launch."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    cxx = os.environ.get("CXX") or shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    from paper_2402_19364_gb300 import build
    build.build()
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    exe = str(tmp_path_factory.mktemp("fake") / "fake_cuda_check")
    objs = [str(obj) for _, obj, _ in build._units()]
    subprocess.run([cxx, "-O1", "-std=c++17", "-Wall", "-I", cuda, "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "fake_cuda_check.cpp"), *objs, "-lpthread", "-o", exe], check=True)

    def run(name):
        out = subprocess.run([exe, name], capture_output=True, text=True, timeout=300)
        assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
    return run


@pytest.mark.parametrize("name", ["retiled_member", "own_barrier_count", "tuned_on_its_device", "failed_retuning"])
def test_host_logic(check, name):
    check(name)
