"""CPU: device arithmetic that needs no GPU, compiled for the host from the kernels' headers."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2011_14984_gb300", "csrc")


def _host_library(tmp_path, source):
    src, lib = tmp_path / "host.cc", tmp_path / "host.so"
    src.write_text("#define __host__\n#define __device__\n#define __forceinline__ inline\n" + source)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", f"-I{CSRC}", str(src),
                    "-o", str(lib)], check=True)
    return ctypes.CDLL(str(lib))


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


@pytest.mark.parametrize("half", [1e-4, 1e-2, 1.0, 30.0])
def test_point_gap_is_a_lower_bound(tmp_path, half):
    # receivers at offsets of up to 50 from their tile's centre, from boxes near them and far: the exact
    # distance (in 64 bits, from the FP32 centres and half sizes) is never below the bound, and the
    # bound is within the margin that it names (2e-6 of the operands a component)
    lib = _host_library(tmp_path, """
#include "tile_bounds.cuh"
extern "C" void gaps(int n, const float *dc, const float *x, const float *h, float *out)
{
    for (int i = 0; i < n; ++i)
        out[i] = frost::gap2(frost::point_axis_gap(dc[3 * i], x[3 * i], h[3 * i]),
                             frost::point_axis_gap(dc[3 * i + 1], x[3 * i + 1], h[3 * i + 1]),
                             frost::point_axis_gap(dc[3 * i + 2], x[3 * i + 2], h[3 * i + 2]));
}
""")
    rng = np.random.default_rng(8)
    n = 200000
    cj = rng.uniform(-1, 1, (n, 3)).astype(np.float32)
    x = rng.uniform(-50, 50, (n, 3))
    # the exact offset from the box's centre: within a few half sizes, or anywhere
    near = half * rng.uniform(-4, 4, (n, 3))
    off = np.where(rng.random((n, 1)) < 0.7, near, rng.uniform(-60, 60, (n, 3)))
    cw = (cj + off - x).astype(np.float32)          # the receivers' tile centres
    x = cj.astype(np.float64) + off - cw            # exact offsets from them
    h = (half * rng.uniform(0.5, 1, (n, 3))).astype(np.float32)
    dc, xh = cw - cj, x.astype(np.float32)
    out = np.empty(n, np.float32)
    lib.gaps(n, _p(np.ascontiguousarray(dc)), _p(np.ascontiguousarray(xh)), _p(h), _p(out))
    exact = np.maximum(0.0, np.abs(off) - h)
    assert np.all(out.astype(np.float64) <= (exact ** 2).sum(axis=1))
    margin = 2e-6 * (np.abs(dc) + np.abs(x) + h)
    least = np.maximum(0.0, exact - margin)
    assert np.all(out >= (least ** 2).sum(axis=1) * (1 - 1e-6))
