"""The library's host side without a GPU: its objects linked with a stand-in for
the CUDA runtime (tests/c/fake_cuda) that keeps, for every device, how much
dynamic shared memory a kernel may use there, and refuses launches beyond it.
Every call runs on two devices of one process, one after the other, and with
searches whose launch fails; and which calls' launches overlap."""
import glob
import importlib.util
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FAKE = os.path.join(ROOT, "tests", "c", "fake_cuda")


@pytest.fixture(scope="module")
def host_check(tmp_path_factory):
    path = os.path.join(ROOT, "paper_2409_05500_gb300", "build.py")
    spec = importlib.util.spec_from_file_location("_vl_build_host", path)
    build = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(build)
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    build.build()
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc())))
    exe = str(tmp_path_factory.mktemp("fake_cuda") / "host_check")
    subprocess.run([gxx, "-O1", "-std=c++17", "-I", FAKE, "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(cuda, "include"), os.path.join(FAKE, "host_check.cpp"),
                    os.path.join(FAKE, "fake_cuda.cpp"),
                    *sorted(glob.glob(os.path.join(build.BUILD, "*.o"))), "-lpthread", "-o", exe],
                   check=True)
    return exe


@pytest.mark.parametrize("what", ["two_devices", "no_search", "overlap"])
def test_host_side(host_check, what):
    out = subprocess.run([host_check, what], check=True, capture_output=True, text=True).stdout
    assert out == ""
