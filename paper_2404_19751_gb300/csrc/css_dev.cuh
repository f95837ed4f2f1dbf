// css_dev.cuh -- device data layout and helpers shared by the library's kernels.
//
// Half-edge convention: face f, corner k, half-edge h = 3f+k runs from corner k to
// corner k+1.  The face layout puts corner 0 at (0,0), corner 1 at (L01,0) and
// corner 2 at (x2, y2 > 0).  The frame of half-edge h has its origin at corner k,
// x along the edge and +y pointing into face f.  A window lives on the half-edge
// of the face it propagates into; its pseudo-source s lies on the other side.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#define CSS_FULL 0xffffffffu

namespace css {

// Per half-edge record (64 B): everything one unfolding step needs.  Lengths are in units of the mesh
// (DMesh::unit).
struct __align__(16) HeRec {
    double L;        // edge length
    double cx, cy;   // opposite corner c in this half-edge frame (cy > 0)
    double cl, sl;   // cos/sin of angle(c): rotation into the frame across edge c-u
    double cr, sr;   // cos/sin of angle(v - c): rotation into the frame across edge v-c
    int32_t tl, tr;  // twin of half-edge (f,k+2) [edge c-u] and (f,k+1) [edge v-c], -1: boundary
};

// FP32 copy of HeRec for the FP32 form's arithmetic (32 B)
struct __align__(16) HeRec32 {
    float L, cx, cy, cl, sl, cr, sr;
    int32_t pad;
};

// Half-edge topology for unfolding (16 B): the vertices at the start, the end and the far corner
// (bit 30: shortest paths may bend there, see EMITS), and the face's rank (bucket index)
constexpr int32_t EMITS = 1 << 30, VMASK = EMITS - 1;

struct DMesh {
    int32_t nv, nf;
    int32_t periodic;
    double per[2];
    // The power of two next below a typical edge length.  he and he32 hold lengths divided by it, which
    // is exact, so that squares of lengths stay in FP32's range whatever the mesh's scale; all other
    // arrays are in the caller's units.
    double unit, inv_unit;
    const HeRec* he;              // 3 nf
    const int32_t* twin;          // 3 nf
    const int32_t* fv;            // 3 nf, vertex at each corner
    const double* lay;            // 3 nf: L01, x2, y2 per face
    const double* frame;          // 9 nf: origin, e1, e2 per face (world)
    const double* theta;          // nv angle sums
    const uint8_t* bnd;           // nv: boundary vertex
    const int32_t* ring_start;    // nv + 1
    const int32_t* ring;          // 3 nf corners h with fv[h] == v, grouped by vertex
    const HeRec32* he32;          // 3 nf, FP32 copies of he
    const int32_t* frank;         // nf: rank of each face along a Morton curve (bucket order)
    const float2* cang;           // 3 nf: (start, width) of corner h around its vertex, angles
                                  // counted counter-clockwise from one fixed edge; NaN on boundary
                                  // and non-manifold vertices
    const int4* htop;             // 3 nf: (start, end, far corner, face rank); vertices that are on the
                                  // boundary, non-manifold or of an angle sum above 2 pi carry EMITS
};

__device__ __forceinline__ void face_corner(const DMesh& m, int f, int k, double& x, double& y) {
    k = (k >= 3) ? k - 3 : k;
    if (k == 0) { x = 0.0; y = 0.0; }
    else if (k == 1) { x = m.lay[3 * f]; y = 0.0; }
    else { x = m.lay[3 * f + 1]; y = m.lay[3 * f + 2]; }
}

__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

template <class T>
__device__ __forceinline__ T warp_sum(T v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(CSS_FULL, v, o);
    return v;
}

// status bits written to the device status word
enum : int {
    ST_WIN_OVERFLOW = 1,     // window pool full
    ST_HASH_OVERFLOW = 2,    // a hash table full
    ST_PAIR_OVERFLOW = 4,    // per-source pair slab full
    ST_ITER_LIMIT = 8,       // loop cap reached
    ST_WALK_LIMIT = 32,      // face walk iteration cap
    ST_BAD_INPUT = 64,
};

}  // namespace css
