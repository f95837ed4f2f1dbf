// geo_common.cuh -- device helpers shared by the neighbour / force kernels.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/css.h"
#include "css_dev.cuh"

namespace geo {

using css::DMesh;

// Widening (rad) of the range in which a shortest path can leave a vertex it passes through.
constexpr float SHADOW_TOL = 1e-3f;

// Cumulative angle at a vertex of the direction g, given the vertex's corner hc whose first
// edge runs along e (both in one face layout); NaN when g is too short to have a reliable
// direction or the corner has no cumulative angle.
__device__ __forceinline__ float back_angle(const DMesh& m, int hc, double ex, double ey, double gx, double gy,
                                            double scale) {
    if (hc < 0 || !(gx * gx + gy * gy > 1e-12 * scale * scale)) return __int_as_float(0x7fffffff);
    return m.cang[hc].x + atan2f((float)(ex * gy - ey * gx), (float)(ex * gx + ey * gy));
}

// A back direction in 16 bits: steps of 1/4096 rad offset by 4 rad; 0xffff where it is unknown or
// out of range.
constexpr float BACK_STEP = 4096.0f, BACK_OFF = 4.0f;
__device__ __forceinline__ unsigned pack_back(float b) {
    const float t = (b + BACK_OFF) * BACK_STEP;
    return (t >= 0.0f && t < 65535.0f) ? (unsigned)__float2int_rn(t) : 0xffffu;   // NaN -> unknown
}
__device__ __forceinline__ float unpack_back(unsigned q) { return (float)q * (1.0f / BACK_STEP) - BACK_OFF; }

__device__ __forceinline__ double pot_dudl(const css_potential& p, double l) {
    if (!(l < p.r_cut)) return 0.0;
    if (p.kind == CSS_POT_HARMONIC) return -2.0 * p.eps * (1.0 - l / p.sigma) / p.sigma;
    if (p.kind == CSS_POT_WCA) {
        const double q = p.sigma / l, q2 = q * q, q6 = q2 * q2 * q2;
        return 24.0 * p.eps * (q6 - 2.0 * q6 * q6) / l;
    }
    return -(l / (p.sigma * p.sigma)) * p.A * exp(-l * l / (2.0 * p.sigma * p.sigma));
}

__device__ __forceinline__ double pot_u(const css_potential& p, double l) {
    if (!(l < p.r_cut)) return 0.0;
    if (p.kind == CSS_POT_HARMONIC) { const double u = 1.0 - l / p.sigma; return p.eps * u * u; }
    if (p.kind == CSS_POT_WCA) {
        const double q = p.sigma / l, q2 = q * q, q6 = q2 * q2 * q2;
        return 4.0 * p.eps * (q6 * q6 - q6) + p.eps;
    }
    return p.A * exp(-l * l / (2.0 * p.sigma * p.sigma));
}

// Inclusive prefix sum of x over the warp.
__device__ __forceinline__ int warp_incl_scan(int x, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(CSS_FULL, x, o);
        if (lane >= o) x += t;
    }
    return x;
}

// The lane whose inclusive-scan range holds item t (31 for t beyond the total).
__device__ __forceinline__ int scan_owner(int incl, int t) {
    int owner = 0;
#pragma unroll
    for (int step = 16; step >= 1; step >>= 1) {
        const int v = __shfl_sync(CSS_FULL, incl, owner + step - 1);
        if (v <= t) owner += step;
    }
    return min(owner, 31);
}

}  // namespace geo
