// Sample positions of a track (kernels.cuh: Track), shared by the light curves and their adjoint.
#pragma once

#include "kernels.cuh"

namespace scint {

// pixel u 2^-64 n and its fraction; n a power of two of at least 2
SCINT_DEV void grid_pixel(unsigned long long u, int n, int& i, float& t) {
    const int shift = __clz(n) + 1;    // 32 - log2 n
    const unsigned hi = (unsigned)(u >> 32);
    i = (int)(hi >> shift);
    t = (float)__funnelshift_l((unsigned)u, hi, 32 - shift) * 0x1.0p-32f;    // the 32 bits below the pixel
}
SCINT_DEV void track_sample(const Track& tr, int s, int n, int& ix, int& iy, float& tx, float& ty) {
    const unsigned long long k = (unsigned)s;
    grid_pixel(tr.x0 + k * tr.dx, n, ix, tx);
    grid_pixel(tr.y0 + k * tr.dy, n, iy, ty);
}

}  // namespace scint
