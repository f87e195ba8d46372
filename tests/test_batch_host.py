"""The host code of batches and serving, built with g++ over a stand-in for the
device (tests/native/batch_host.cpp): the states that a real kernel reports only
when something went wrong are set by hand there."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    from paper_1306_1467_gb300 import build
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc())))
    include = next((d for d in (os.path.join(cuda, "include"), os.path.join(cuda, "targets", "x86_64-linux", "include"))
                    if os.path.exists(os.path.join(d, "cuda_runtime.h"))), None)
    if include is None or shutil.which("g++") is None:
        pytest.skip("needs g++ and the CUDA headers")
    out = str(tmp_path_factory.mktemp("native") / "batch_host")
    r = subprocess.run(["g++", "-std=c++17", "-O1", "-g", "-D_GLIBCXX_ASSERTIONS", "-x", "c++", "-pthread", "-I", include,
                        "-I", os.path.join(ROOT, "include"), "-I", build.CSRC,
                        os.path.join(ROOT, "tests", "native", "batch_host.cpp"), "-o", out], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return out


@pytest.mark.parametrize("case", ["flags", "step_counts"])
def test_batch_host(program, case):
    r = subprocess.run([program, case], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "ok", r.stdout + r.stderr
