"""Host code of the library on the CPU: csrc/fdtd_capi.cu is compiled into
tests/host_runtime.cpp, whose CUDA runtime keeps device memory on the host and
runs queued work as late as a stream may (see there)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1008_2602_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(CUDA_INC, "cuda.h")):
        pytest.skip("g++ and the CUDA headers are needed to compile the host code")
    exe = tmp_path_factory.mktemp("host") / "host_runtime"
    subprocess.run([gxx, "-std=c++17", "-O1", "-fopenmp", "-Wno-unknown-pragmas", "-I", CSRC, "-I", CUDA_INC, "-o", str(exe),
                    os.path.join(ROOT, "tests", "host_runtime.cpp"), "-ldl"], check=True)
    return str(exe)


@pytest.mark.parametrize("scenario", ["factors", "refused", "chosen", "split", "segments", "waits", "checkpoint", "memory"])
def test_host_code(program, scenario):
    r = subprocess.run([program, scenario], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
