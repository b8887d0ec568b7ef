"""The fill's kernel under every order in which a block's warps may be
scheduled late: its source runs on the CPU with one warp held back to the last
moment, and the surface is compared with the oracle bit for bit.  (A warp that
reads the tile's record after another has cleared it leaves its part of the
tile unread.)"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
from paper_2606_12800_gb300 import inputs

HERE = os.path.dirname(os.path.abspath(__file__))
FILL = os.path.join(os.path.dirname(HERE), "paper_2606_12800_gb300", "csrc", "fr_fill.cu")

DRIVER = r"""
#include "simt.h"
namespace {
%s
}
extern "C" void sweep(const float* z, int64_t nx, int64_t ny, float* F, uint8_t* act, uint8_t* next, int first,
                      int passes, int late, unsigned long long* changed) {
    const unsigned tiles = (unsigned)(((nx + kFT - 1) / kFT) * ((ny + kFT - 1) / kFT));
    for (blockIdx.x = 0; blockIdx.x < tiles; ++blockIdx.x)
        simt::run_block(kFNT, late, [&] {
            if (first) k_fill_sweep<true>(z, nx, ny, F, act, next, passes, changed);
            else k_fill_sweep<false>(z, nx, ny, F, act, next, passes, changed);
        });
}
"""


@pytest.fixture(scope="module")
def kernel(tmp_path_factory):
    src = open(FILL).read()
    begin = src.index("constexpr int kFT ")
    src = src[begin:src.index("}  // namespace", begin)]
    d = tmp_path_factory.mktemp("fill")
    cpp, so = str(d / "fill.cpp"), str(d / "fill.so")
    with open(cpp, "w") as f:
        f.write(DRIVER % src)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I" + HERE, cpp, "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("late", range(-1, 8))
def test_fill_with_a_late_warp(kernel, late):
    ny, nx = 70, 197
    z = inputs.fractal_dem(ny, nx, beta=2.2, tilt=0.0, seed=3)
    F = np.zeros_like(z)
    tiles = ((nx + 63) // 64) * ((ny + 63) // 64)
    act = [np.zeros(tiles, np.uint8), np.zeros(tiles, np.uint8)]
    P = ctypes.c_void_p
    for s in range(1000):
        changed = ctypes.c_uint64(0)
        kernel.sweep(P(z.ctypes.data), ctypes.c_int64(nx), ctypes.c_int64(ny), P(F.ctypes.data),
                     P(act[(s + 1) & 1].ctypes.data), P(act[s & 1].ctypes.data), int(s == 0), 2, late,
                     ctypes.byref(changed))
        if not changed.value:
            break
    np.testing.assert_array_equal(F, oracle.fill(z))
