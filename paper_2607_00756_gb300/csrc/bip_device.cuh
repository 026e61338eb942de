// Device helpers shared by several kernels of the map path.
#pragma once

#include <cuda_runtime.h>

// One axis of the crop mask: the minimum-image offset of the scan at r from
// the site at t lies in [-n/(2f), n/(2f)).  FP64 so the decision matches a
// host FP64 evaluation of the same formula.
__device__ __forceinline__ bool in_crop_axis(double r, double t, int n, int f) {
    double d = r - t;
    d -= n * floor((d + 0.5 * n) / n);
    const double h = 0.5 * n / f;
    return d >= -h && d < h;
}

// Crop mask of Sec. 2.2.4: a site at pixel position (ty, tx) contributes to
// the scan at (ry, rx) when that holds on both axes.
__device__ __forceinline__ bool in_crop(double ry, double rx, double ty, double tx, int ny, int nx, int fy,
                                        int fx) {
    return in_crop_axis(ry, ty, ny, fy) && in_crop_axis(rx, tx, nx, fx);
}

// x mod n in [0, n) for any sign of x (grid lengths need not be powers of
// two: 3 M lengths are allowed).
__device__ __forceinline__ int wrap_n(int x, int n) {
    if ((n & (n - 1)) == 0) return x & (n - 1);   // a power of two: a mask (two's complement)
    const int r = x % n;
    return r < 0 ? r + n : r;
}
