"""The library's device memory (csrc/memory.cu) against a fake CUDA runtime
(memory_fake.cpp), on the host: when a freed block is handed out again,
how much is kept, that threads do not wait for each other's frees,
that nothing kept outlives its context, and that it can be given back."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2302_05662_gb300", "csrc")


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    out = str(tmp_path_factory.mktemp("memory") / "memory_fake")
    subprocess.run(["g++", "-O1", "-g", "-std=c++17", "-pthread", "-I", include, "-I", CSRC, "-x", "c++",
                    os.path.join(CSRC, "memory.cu"), os.path.join(ROOT, "tests", "memory_fake.cpp"), "-o", out], check=True)
    return out


@pytest.mark.parametrize("scenario", ["reuse", "failed_wait", "bounded", "threads", "reset", "trim"])
def test_scenario(program, scenario):
    r = subprocess.run([program, scenario], capture_output=True, text=True, timeout=20)
    assert r.returncode == 0, r.stdout
