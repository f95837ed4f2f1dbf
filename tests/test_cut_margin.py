"""The neighbour kernel's cut of a window by an end vertex's distance, compiled for the host and
compared with FP64: what it cuts has to be reached no later along the edge, whatever the rounding of
its single-precision arguments."""
import ctypes as C
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r"""
#include <cmath>
#define __device__
#define __forceinline__ inline
static inline float __fdividef(float a, float b) { return a / b; }
using std::fmaf;
%s
extern "C" void cuts(long n, const float* sx, const float* s2, const float* a, const float* L, const float* eps, float* out) {
    for (long i = 0; i < n; ++i) out[i] = cut_at(sx[i], s2[i], a[i], L[i], eps[i]);
}
"""


@pytest.fixture(scope="module")
def cuts(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not found")
    src = open(os.path.join(ROOT, "paper_2404_19751_gb300", "csrc", "waves.cu")).read()
    body = re.search(r"^__device__ __forceinline__ float cut_at\(.*?^}", src, re.M | re.S).group(0)
    d = tmp_path_factory.mktemp("cut")
    (d / "cut.cpp").write_text(SHIM % body)
    subprocess.run([gxx, "-O1", "-ffp-contract=off", "-shared", "-fPIC", "-o", str(d / "cut.so"), str(d / "cut.cpp")], check=True)
    lib = C.CDLL(str(d / "cut.so"))

    def run(*args):
        args = [np.ascontiguousarray(x, np.float32) for x in args]
        out = np.empty(len(args[0]), np.float32)
        lib.cuts(C.c_long(len(out)), *[x.ctypes.data_as(C.POINTER(C.c_float)) for x in args + [out]])
        return out
    return run


def _toward_zero(x):
    y = x.astype(np.float32)
    return np.where(np.abs(y.astype(np.float64)) > np.abs(x), np.nextafter(y, np.float32(0)), y)


@pytest.mark.parametrize("end", [0, 1])
def test_cut_parts_are_reached_along_the_edge(cuts, end):
    rng = np.random.default_rng(3)
    n = 1_000_000
    L = rng.uniform(1.0, 2.0, n)
    # pseudo-sources near the edge's line, before and beyond the vertex; its distance less sigma is
    # smaller than the straight one, by as little as rounding and by much
    t = 10.0 ** rng.uniform(-7, 1, n) * rng.choice([-1.0, -1.0, 1.0], n)
    d = 10.0 ** rng.uniform(-10, -1, n)
    sy = -np.sqrt(2.0 * d * 10.0 ** rng.uniform(-4, 4, n))
    far = np.hypot(t, sy)
    a = np.minimum(np.where(t < 0, np.abs(t) + d, far), far * (1.0 - 10.0 ** rng.uniform(-15, -0.5, n)))
    # the kernel's arguments: the frame's coordinate, rounded toward zero, measured from the edge's
    # start or subtracted from its length
    f32 = np.float32
    fx, fy, fl = _toward_zero(t if end == 0 else L - t), _toward_zero(sy), L.astype(f32)
    eps = f32(4.8e-7) * (np.abs(fx) + fl)
    sx = fx if end == 0 else fl - fx
    x0 = cuts(sx, sx * sx + fy * fy, _toward_zero(a), fl, eps).astype(np.float64)
    cut = x0 > 0
    assert cut.mean() > 0.1
    x = np.minimum(x0, L)
    gain = (x + a) - np.hypot(x - t, sy)   # by how much the window beats the way along the edge
    bad = cut & (gain > 1e-14)
    assert not bad.any(), f"{bad.sum()} of {cut.sum()} cut too far, by up to {gain[bad].max()} of an edge"
