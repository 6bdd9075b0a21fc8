// Lower bounds on distances from boxes (centre and half size by component, FP32), for the tile
// kernels of force_tiles.cu.  Every bound holds for the exact positions: the margins cover the
// FP32 evaluation and the rounding of the half sizes and of the receivers' offsets.
#pragma once

#include <cmath>

namespace frost {

// of two intervals whose centres are d apart, with half sizes h in all: the gap is good to a few units
// whatever the distance of the tiles from the origin
__host__ __device__ __forceinline__ float axis_gap(float d, float h)
{
    return fmaxf(0.f, fmaf(fabsf(d), 0.999999f, -1.000001f * h));
}

// of a point at x from the centre of its own tile, dc from the interval's centre.  dc + x cancels
// where a wide tile reaches to the interval, so the margin is of the size of dc and x, not of
// their sum (it is 1e-6 of it; the roundings are below 1.5e-7)
__host__ __device__ __forceinline__ float point_axis_gap(float dc, float x, float h)
{
    return fmaxf(0.f, fmaf(-1e-6f, fabsf(dc) + fabsf(x) + h, fabsf(dc + x) - h));
}

__host__ __device__ __forceinline__ float gap2(float gx, float gy, float gz) { return fmaf(gx, gx, fmaf(gy, gy, gz * gz)); }

}  // namespace frost
