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
