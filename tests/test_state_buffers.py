"""Which buffers lbm_save_state and lbm_load_state may hand to a kernel: memory
of the context's own GPU and managed memory.  A buffer on another GPU (a program
with several replicas) or in host memory goes through cudaMemcpyAsync, since a
kernel that touched it would fault.  The rule is compiled as plain C++; the
source is checked to ask it wherever a caller's state buffer meets a kernel."""
import os
import re
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2203_01316_gb300", "csrc")
UNREGISTERED, HOST, DEVICE, MANAGED = range(4)  # cudaMemoryType


def test_kernels_touch_only_memory_of_their_own_gpu(tmp_path):
    from paper_2203_01316_gb300.build import nvcc
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc()))), "include")
    if not os.path.exists(os.path.join(cuda, "cuda_runtime_api.h")):
        pytest.skip("no CUDA headers")
    exe = str(tmp_path / "reach")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", cuda, os.path.join(HERE, "host", "reach.cpp"), "-o", exe],
                   check=True)
    cases = [(t, of, d) for t in range(4) for of in (0, 1) for d in (0, 1)]
    out = subprocess.run([exe], input="\n".join("%d %d %d" % c for c in cases), check=True, capture_output=True,
                         text=True).stdout.split()
    assert [int(v) for v in out] == [int(t == MANAGED or (t == DEVICE and of == d)) for t, of, d in cases]


def test_state_kernels_ask_for_it():
    src = open(os.path.join(CSRC, "lbm_api.cu")).read()
    for condition in (r"const bool direct = ([^;]*);", r"if \(([^{]*need <= kSmallState[^{]*)\) \{"):
        found = re.findall(condition, src)
        assert found and all("own_memory(c, " in f for f in found)
