"""The node stacks of the warp and block traversals, executed on the CPU: no tree of up to 100 levels
fills them, however many of its nodes are near."""
import ctypes
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
SRC = os.path.join(HERE, "host_exec", "stack_host.cu")
LIB = os.path.join(HERE, "host_exec", "_build", "libstack_host.so")


@pytest.fixture(scope="module")
def walk():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    os.makedirs(os.path.dirname(LIB), exist_ok=True)
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"),
                        SRC, "-o", LIB], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    f = ctypes.CDLL(LIB).hx_stack_walk
    f.restype = ctypes.c_longlong
    f.argtypes = [ctypes.c_int] * 5
    return f


# (nodes a step, entries) of k_wide3, k_rtrav_warp and k_rtrav2
@pytest.mark.parametrize("width,cap", [(32, 768), (32, 2048), (256, 4096)])
@pytest.mark.parametrize("spine,depth", [(0, 1), (0, 5), (0, 26), (20, 20), (85, 14)])
@pytest.mark.parametrize("first", [0, 1])
def test_stacks_hold_every_near_node(walk, width, cap, spine, depth, first):
    assert walk(spine, depth, first, width, cap) == (spine + 2) * 2 ** depth
