"""The library's host code that no entry point reaches by itself (tests/native/host_checks.cpp, linked with the library's
objects): no GPU."""
import os
import subprocess

import pytest

from paper_1911_05146_b200 import build as lib_build

HERE = os.path.dirname(os.path.abspath(__file__))
CUDA = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
WRAPPED = ["cudaGetDevice", "cudaFuncSetAttribute", "cudaGetDriverEntryPoint"]


@pytest.fixture(scope="module")
def checks(tmp_path_factory):
    lib_build.build()
    objects = [os.path.join(lib_build.CSRC, s[:-3] + ".o") for s in lib_build.SOURCES]
    if not all(os.path.exists(o) for o in objects):
        lib_build.build(force=True)
    exe = str(tmp_path_factory.mktemp("native") / "host_checks")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", lib_build.CSRC, "-I", os.path.join(CUDA, "include"),
                    os.path.join(HERE, "native", "host_checks.cpp"), *[o for o in objects if not o.endswith("hpf_model.o")], "-o", exe, "-L", os.path.join(CUDA, "lib64"), "-lcudart", "-lpthread",
                    "-Wl,-rpath," + os.path.join(CUDA, "lib64"), *["-Wl,--wrap=" + f for f in WRAPPED]], check=True, timeout=300)
    return exe


@pytest.mark.parametrize("name", ["attributes_per_device", "cells_are_planned_for_one_micro_batch", "launches_cover_all_micro_batches", "calls_by_themselves",
                                  "weight_gradients_of_a_step"])
def test_host(checks, name):
    r = subprocess.run([checks, name], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr
