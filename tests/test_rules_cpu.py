"""The library's host-side choices, compiled alone with the host compiler (no
GPU, no library)."""
import ctypes
import os
import subprocess
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_12707_gb300", "csrc")


def compile_host(path, source, *files):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    src, lib = os.path.join(path, "shim.cpp"), os.path.join(path, "shim.so")
    with open(src, "w") as f:
        f.write(textwrap.dedent(source))
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, "-I", os.path.join(cuda, "include"),
                    src, *(os.path.join(CSRC, x) for x in files), "-o", lib], check=True)
    return ctypes.CDLL(lib)


def test_setup_runs_once_on_each_device(tmp_path):
    """A kernel attribute holds on the device it was set on: the second device
    gets its own call, a failed one is tried again."""
    lib = compile_host(str(tmp_path), """
        #include "kvd_internal.h"
        static kvd::OncePerDevice once;
        static int calls[128];
        extern "C" int setup(int device, int result)
        {
            return once(device, [&] { ++calls[device]; return (cudaError_t)result; });
        }
        extern "C" int count(int device) { return calls[device]; }
    """)
    assert [lib.setup(0, 0), lib.setup(0, 0), lib.setup(1, 0), lib.setup(0, 0), lib.setup(1, 0)] == [0] * 5
    assert [lib.count(0), lib.count(1)] == [1, 1]
    assert [lib.setup(2, 1), lib.setup(2, 0), lib.setup(2, 1)] == [1, 0, 0] and lib.count(2) == 2
    assert [lib.setup(100, 0), lib.setup(100, 0)] == [0, 0] and lib.count(100) == 2   # past the table: every time
