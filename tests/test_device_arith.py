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
    (tmp_path / "cuda_runtime.h").write_text("")
    src.write_text("#define __host__\n#define __device__\n#define __forceinline__ inline\n" + source)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-shared", "-fPIC", f"-I{tmp_path}", f"-I{CSRC}",
                    str(src), "-o", str(lib)], check=True)
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


def test_integer_conversions_are_the_casts(tmp_path):
    # the bits of (double)f and (float)d: FP32 values over all exponents and signs, FP64 values around
    # every exponent of the FP32 range with the fractions that decide a rounding (ties to even both
    # ways, one unit to either side, carries into the next exponent), zeros, the normal range's ends
    lib = _host_library(tmp_path, """
#include <cmath>
#include <cstdint>
#include <cstring>
static unsigned __float_as_uint(float f) { unsigned u; std::memcpy(&u, &f, 4); return u; }
static float __uint_as_float(unsigned u) { float f; std::memcpy(&f, &u, 4); return f; }
static double __hiloint2double(int hi, int lo)
{
    const uint64_t u = ((uint64_t)(unsigned)hi << 32) | (unsigned)lo;
    double d; std::memcpy(&d, &u, 8); return d;
}
static int __double2hiint(double d) { uint64_t u; std::memcpy(&u, &d, 8); return (int)(u >> 32); }
static int __double2loint(double d) { uint64_t u; std::memcpy(&u, &d, 8); return (int)u; }
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fmul_rn(float a, float b) { return a * b; }
static float rsqrtf(float a) { return 1.f / std::sqrt(a); }
#include "df_arith.cuh"
extern "C" void to_double(int n, const float *f, double *d) { for (int i = 0; i < n; ++i) d[i] = frost::df::f2d(f[i]); }
extern "C" void to_float(int n, const double *d, float *f) { for (int i = 0; i < n; ++i) f[i] = frost::df::d2f(d[i]); }
""")
    rng = np.random.default_rng(9)
    expo = np.arange(256, dtype=np.uint32)
    frac = np.concatenate([[0, 1, 2, 0x3fffff, 0x400000, 0x7ffffe, 0x7fffff],
                           rng.integers(0, 1 << 23, 249)]).astype(np.uint32)
    bits = ((expo[:, None] << 23) | frac[None, :]).ravel()
    bits = np.concatenate([bits, bits | np.uint32(0x80000000)])
    f = np.ascontiguousarray(bits).view(np.float32)
    d = np.empty(f.size)
    lib.to_double(f.size, _p(f), _p(d))
    with np.errstate(invalid="ignore"):
        r = f.astype(np.float64)
    assert np.array_equal(d, r, equal_nan=True) and np.array_equal(np.signbit(d), np.signbit(r))

    expo = np.concatenate([np.arange(880, 1170), [0, 1, 2046, 2047]]).astype(np.uint64)
    high = np.concatenate([[0, 1, 2, (1 << 23) - 2, (1 << 23) - 1], rng.integers(0, 1 << 23, 59)]).astype(np.uint64)
    low = np.concatenate([[0, 1, (1 << 28) - 1, 1 << 28, (1 << 28) + 1, (1 << 29) - 1],
                          rng.integers(0, 1 << 29, 26)]).astype(np.uint64)
    bits = ((expo[:, None, None] << np.uint64(52)) | (high[None, :, None] << np.uint64(29)) | low[None, None, :]).ravel()
    bits = np.concatenate([bits, bits | np.uint64(1 << 63)])
    d = np.ascontiguousarray(bits).view(np.float64)
    f = np.empty(d.size, np.float32)
    lib.to_float(d.size, _p(d), _p(f))
    with np.errstate(over="ignore", invalid="ignore"):
        r = d.astype(np.float32)
    assert np.array_equal(f, r, equal_nan=True) and np.array_equal(np.signbit(f), np.signbit(r))
