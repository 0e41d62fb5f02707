"""The network context's set-up on CPU (no GPU): the library's host code with
the CUDA runtime's calls replaced by fakes (tests/host/kp_mlp_harness.cu)."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "tests", "host", "kp_mlp_harness.cu")
OUT = os.path.join(ROOT, "tests", "host", "_build", "libkphostmlp.so")
CSRC = os.path.join(ROOT, "paper_2409_06807_gb300", "csrc")


@pytest.fixture(scope="module")
def H():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc is needed to build the host harness")
    deps = [SRC, os.path.join(ROOT, "include", "kp.h")] + \
        [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    if not os.path.exists(OUT) or any(os.path.getmtime(p) > os.path.getmtime(OUT) for p in deps):
        os.makedirs(os.path.dirname(OUT), exist_ok=True)
        tmp = OUT + f".tmp{os.getpid()}"
        subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17",
                        "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"),
                        "-o", tmp, SRC, "-cudart", "static"], check=True)
        os.replace(tmp, OUT)
    return C.CDLL(OUT)


def test_every_device_gets_the_shared_memory_limit(H):
    """The limit of a kernel's dynamic shared memory belongs to a device: a
    network created on a second one in the same process sets it there too."""
    for device in (0, 1, 0, 3):
        H.kpt_mlp_create_on(device)
        for training in (0, 1):
            assert H.kpt_mlp_limit(device, training) == H.kpt_mlp_needs(training) > 48 * 1024
