"""The FP64 sum of 2D leaf angles, executed on the CPU, where leaves are seen under exactly or
nearly 45 degrees."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
SRC = os.path.join(HERE, "host_exec", "angle64_host.cu")
LIB = os.path.join(HERE, "host_exec", "_build", "libangle64_host.so")


@pytest.fixture(scope="module")
def hx():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    os.makedirs(os.path.dirname(LIB), exist_ok=True)
    r = subprocess.run([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a", "-Xcompiler",
                        "-fPIC,-ffp-contract=off", "-shared", "-I", os.path.join(ROOT, "include"), SRC, "-o", LIB],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    f = ctypes.CDLL(LIB).hx_angle64
    f.restype = ctypes.c_double
    f.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_double, ctypes.c_double, ctypes.c_int]

    def run(p, q, stride=1):
        p = np.ascontiguousarray(p)
        return f(p.ctypes.data, len(p), float(q[0]), float(q[1]), stride)
    return run


def _loop(shape, c, r, copies):
    """Eight leaves around c, each `copies` times in a row: a square with halved sides or a circle's arcs."""
    v = np.array([[1, 0], [1, 1], [0, 1], [-1, 1], [-1, 0], [-1, -1], [0, -1], [1, -1]], dtype=float)
    if shape == "circle":
        t = 0.25 * np.pi * np.arange(8)
        v = np.stack([np.cos(t), np.sin(t)], axis=1)
    v = c + r * v
    return np.repeat(np.concatenate([v, np.roll(v, -1, axis=0)], axis=1), copies, axis=0)


@pytest.mark.parametrize("copies,stride", [(1, 1), (32, 1), (32, 32)])
@pytest.mark.parametrize("ccw", [True, False])
@pytest.mark.parametrize("shape", ["square", "circle"])
def test_leaves_of_45_degrees(hx, shape, ccw, copies, stride):
    """At the centre the sum is a whole number of turns: 8 copies angles, each rounded to 2^-52 of
    it, 1e-13 for 256 of them."""
    rng = np.random.default_rng(3)
    for k in range(300):
        c = np.zeros(2) if k == 0 else rng.uniform(-1, 1, 2)
        p = _loop(shape, c, 1.0 if k == 0 else np.exp(rng.uniform(-2, 2)), copies)
        if not ccw:
            p = p[::-1][:, [2, 3, 0, 1]]
        assert abs(hx(p, c, stride) - (copies if ccw else -copies)) <= 1e-13 * copies


@pytest.mark.parametrize("e", range(-75, 80, 5))
def test_scales(hx, e):
    """A closed loop of 24 leaves of 15 degrees at any scale that one arc tangent per leaf holds
    (products of coordinates above 1e-300 and below 1e300): one turn inside, none outside, to the
    leaves' rounding (24 x 2^-52)."""
    t = 2 * np.pi * np.arange(24) / 24
    v = 10.0 ** e * np.stack([np.cos(t), np.sin(t)], axis=1)
    p = np.concatenate([v, np.roll(v, -1, axis=0)], axis=1)
    for q, w in (((0.0, 0.0), 1.0), ((0.3, -0.2), 1.0), ((3.0, 1.0), 0.0), ((1e3, 2e3), 0.0)):
        assert abs(hx(p, 10.0 ** e * np.array(q)) - w) <= 1e-14
