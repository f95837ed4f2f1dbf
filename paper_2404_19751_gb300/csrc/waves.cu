// waves.cu -- cutoff geodesic neighbours and forces by window propagation without window lists.
//
// Method (Sec. 2.2 and Sec. 3.1 of the paper).  A window is the part of an edge that straight
// lines from a pseudo-source s (the source, or a boundary or saddle vertex where shortest paths
// bend) reach through the faces unfolded so far; it carries the length sigma + |x - s|, sigma
// being the length from the source to s.  Unfolding a window into the next face gives a
// candidate for the distance of the face's far corner and at most two child windows.
// Windows are never compared with one another.  Each is cut by the distances of its edge's two
// end vertices only: the part of the edge that the path through an end vertex and along the
// edge reaches no later is dropped (the filter of Xin and Wang, "Improving Chen and Han's
// algorithm on the discrete geodesic problem", ACM TOG 2009, in the form of an interval).  A
// vertex distance is the length of a real path, so what is dropped is no part of a shortest
// path, and what remains still holds every shortest path.  A vertex starts windows of its own
// once its distance is final (no waiting window has a smaller key), and only into the wedge in
// which a shortest path through it can continue.
//
// Since nothing compares windows, nothing keeps them: a window is needed from the wave that
// makes it to the wave that unfolds it.  The waiting windows are a first-in first-out ring in
// shared memory, the only other state is the table of vertex distances, and a wave is 32
// windows whatever their keys (measured on the workloads: taking the smallest keys first
// unfolds no fewer windows than the order of creation).  The particles of a face are tested
// against each window that enters it; the tests are queued and evaluated when ten are there.
//
// A window's cone is two directions in the frame of its pseudo-source, where they stay what
// they are through every unfolding (the direction to the vertex that bounds the cone), so no
// error builds up and no ray has to be cut with an edge in FP64: the interval on the edge is
// FP32 and rounded outward.  Windows are the same in both forms, FP64 images, rotations and rims:
// with a rotation of its own in FP32, each of the two children of a corner drifts by 6e-8 of a turn
// an unfolding, and behind a flat vertex nothing covers the gap between them (100 of 6 M pairs of a
// flat sheet of 80 x 80 vertices were lost, 1270 of 4 M at 200 x 200; with FP32 rims alone 1 of 6 M).
// The FP32 form tests its targets and keeps the directions of paths in FP32; lengths of results are
// FP64 in both forms.  All lengths in this file are in units of the mesh (DMesh::unit), so the FP32
// filters and roots see the same numbers at every scale; results are multiplied back, exactly.
//
// Measured against windows kept in per-edge lists and trimmed against one another (the same
// calls, default launch shapes): 65536 particles on a noisy level-8 sphere 110.7 -> 10.1 ms
// (FP64) and 73.1 -> 10.3 ms (FP32), 8192 on a 256 x 256 height field 130-166 -> 8.3 ms, every pair
// of 64 on a flat plane 27 -> 0.66 ms.  The windows unfolded per source are the same within 10 %
// (482 against 440, 3991 against 3950, 5135 against 5151).
#include <cuda_runtime.h>
#include <limits.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include <math_constants.h>

#include "css_internal.h"
#include "geo_common.cuh"

namespace {

using css::DMesh;
using css::HeRec;
using cssi::WaveLay;
using cssi::WaveWs;

// Where sources fill the chip, instruction fetch sets the pace: a wave is about 2000 instructions of
// mostly straight code, 16 warps sit at different places of it, and 43 % of stall cycles waited for
// instructions.  So loops are not unrolled, rare branches are marked and divisions in FP32 are the
// short ones (16384 sources on a noisy sphere: 2.96 -> 2.45 ms in FP64; 2048 on a 128 x 128 height field
// 3.55 -> 3.23; small sets and teams unchanged within 2 %).
constexpr int MAXW = 8;          // warps per CTA
constexpr int EV = 10;           // queued target tests per warp
constexpr int NONE = -1;
constexpr int FIRST = 1 << 30;   // ring entry: starts at a vertex of the face behind its edge
constexpr int FROM_VERTEX = 1 << 29;   // test: straight from a vertex of the target's face
constexpr unsigned QUEUED = 1u << 31;  // path record: its vertex waits to start windows

template <class R>
struct Vec2;
template <>
struct Vec2<double> {
    using type = double2;
};
template <>
struct Vec2<float> {
    using type = float2;
};
template <class R>
using V2 = typename Vec2<R>::type;
__device__ __forceinline__ double2 vec2(double x, double y) { return make_double2(x, y); }
__device__ __forceinline__ float2 vec2(float x, float y) { return make_float2(x, y); }

// index of a vertex slot or of a vertex's path record: 16 bits where the tables are in shared memory
template <int PL>
struct Index;
template <>
struct Index<1> {
    using type = uint16_t;
    using pair = ushort2;
    static constexpr uint16_t none = 0xffffu;
    static __device__ __forceinline__ ushort2 make(int a, int b) { return make_ushort2((uint16_t)a, (uint16_t)b); }
};
template <>
struct Index<0> {
    using type = int32_t;
    using pair = int2;
    static constexpr int32_t none = -1;
    static __device__ __forceinline__ int2 make(int a, int b) { return make_int2(a, b); }
};

// a corner within this of a rim does not split the cone (relative to its distance)
constexpr double RIM_MIN = 1e-12;
// tolerance of a point on the rim of a cone, relative to its distance (FP32: the roundings of the
// target's point, the rotation and the rim add up to 6.5e-7 at most)
template <class R>
struct Rim;
template <>
struct Rim<double> {
    static constexpr double t = 4e-12;
};
template <>
struct Rim<float> {
    static constexpr float t = 2e-6f;
};
// FP32 form: relative excess up to which a window's path is taken over a path from a vertex of the
// target's face
constexpr double TIE32 = 1e-6;

// the counters of one source
struct GroupSm {
    int head, tail;      // first waiting window and end of the ring (both only grow)
    int shead, stail;    // the same of the spill area
    int nem[2], cur;     // vertices waiting to start windows: two lists, the one in use
    unsigned emin;       // a lower bound on their distances (FP32 bits)
    int nv, ni, nt, nlog;   // table entries: vertices, their path records, targets, improvements
    int err;
    int item;
};
// a team's per-warp values
struct TeamSm {
    float km[MAXW];
    double fx[MAXW], fy[MAXW], en[MAXW];
};

// ------------------------------------------------------------------ links of paths
// How a vertex or a target was reached (LK instantiations, FP64, one warp per source): the slot of
// the vertex its last straight leg comes from (NONE: the source), and the leg back, as a unit
// direction and a length, in the layout of face fk / 4 from its corner fk % 4 (3: from the target).
// In global memory behind the group's spill area, the vertices' links, then the targets': they are
// written on improvements only and read once per leg.
struct Link {
    int par, fk;
    double len;
    double2 dir;
};
template <bool LK>
struct Links {};
template <>
struct Links<true> {
    Link* p;
};

// corner k of face f in its layout, in units of the mesh
__device__ __forceinline__ void unit_corner(const DMesh& m, int f, int k, double& x, double& y) {
    css::face_corner(m, f, k, x, y);
    x *= m.inv_unit;
    y *= m.inv_unit;
}

// the link of the point (X, Y) of half-edge he's frame straight back to the pseudo-source S: which
// 2 the far corner of the face the window enters, 3 a point in that face; 0, 1 the start and the end of
// the edge, whose leg points into the face on the other side and is written in that face
__device__ __forceinline__ void link_back(const DMesh& m, int he, double2 S, double X, double Y, int which, int par, Link& l) {
    const double a = S.x - X, b = S.y - Y, n = sqrt(a * a + b * b);
    double va = n > 0.0 ? a / n : 1.0, vb = n > 0.0 ? b / n : 0.0;
    int g = he / 3, kg = he - 3 * g, kc = which == 2 ? (kg == 0 ? 2 : kg - 1) : 3;
    if (which < 2 && m.twin[he] >= 0) {
        const int tw = m.twin[he];   // runs from the edge's end to its start
        g = tw / 3;
        kg = tw - 3 * g;
        kc = which == 0 ? (kg == 2 ? 0 : kg + 1) : kg;
        va = -va;
        vb = -vb;
    }
    double ax, ay, bx, by;
    unit_corner(m, g, kg, ax, ay);
    unit_corner(m, g, kg + 1, bx, by);
    const double L = sqrt((bx - ax) * (bx - ax) + (by - ay) * (by - ay));
    const double ex = (bx - ax) / L, ey = (by - ay) / L;
    l.par = par;
    l.fk = 4 * g + kc;
    l.len = n;
    l.dir = make_double2(va * ex - vb * ey, va * ey + vb * ex);
}

// ------------------------------------------------------------------ working memory
template <class T>
__device__ __forceinline__ T* at(unsigned char* b, int off) { return reinterpret_cast<T*>(b + off); }

__device__ __forceinline__ uint32_t hash_of(int32_t key, int logcap) { return ((uint32_t)key * 2654435761u) >> (32 - logcap); }

// slot of the key, claimed if it is new; NONE when the table holds `most` keys already
__device__ __forceinline__ int tab_insert(int32_t* keys, int logcap, int32_t key, int* count, int most, bool& claimed) {
    const uint32_t mask = (1u << logcap) - 1u;
    uint32_t s = hash_of(key, logcap);
    claimed = false;
#pragma unroll 1
    for (uint32_t p = 0; p <= mask; ++p) {
        const int32_t c = *(volatile int32_t*)(keys + s);
        if (c == key) return (int)s;
        if (c == NONE) {
            if (*(volatile int*)count >= most) return NONE;
            const int32_t prev = atomicCAS(keys + s, NONE, key);
            if (prev == NONE) {
                atomicAdd(count, 1);
                claimed = true;
                return (int)s;
            }
            if (prev == key) return (int)s;
        }
        s = (s + 1u) & mask;
    }
    return NONE;
}

// FP64 instructions run at 1/58 of the FP32 rate, conversions among them, and were what bounded the
// FP64 form with 16 warps on an SM (about 130 a wave; 46 with these conversions, FP32 tests of the
// rims and the roots below: 4.03 -> 2.95 ms for 16384 sources on a noisy sphere, 0.27 -> 0.14 ms
// for 1024 on an icosphere).  So values only needed to FP32 precision are converted with integer
// instructions, rounded toward zero: too small becomes 0, too large the largest number.
__device__ __forceinline__ float f32(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned mag = min(hi & 0x7fffffffu, 0x47efffffu);
    const unsigned f = __funnelshift_l(lo, mag - 0x38000000u, 3);
    return __uint_as_float((mag < 0x38100000u ? 0u : f) | (hi & 0x80000000u));
}
__device__ __forceinline__ float f32(float x) { return x; }
__device__ __forceinline__ double f64(float x) {   // x > 0 and normal
    const unsigned f = __float_as_uint(x);
    return __hiloint2double((int)((f >> 3) + 0x38000000u), (int)(f << 29));
}
template <class R>
__device__ __forceinline__ V2<R> narrow(double2 v) {
    if constexpr (sizeof(R) == 8) return v;
    else return make_float2(f32(v.x), f32(v.y));
}
// square root to 2^-22
__device__ __forceinline__ float root(float x) { return x > 0.0f ? x * rsqrtf(x) : 0.0f; }
// x^(1/2) and x^(-1/2) in FP64 from the FP32 reciprocal root: Goldschmidt's iteration (it squares the
// relative error: 2^-22, 2^-43), then a Newton step each on the residual; x normal in FP32
__device__ __forceinline__ void roots(double x, double& r, double& inv) {
    const double y = f64(rsqrtf(f32(x)));
    double g = x * y, h = 0.5 * y;
    const double e = fma(-g, h, 0.5);
    g = fma(g, e, g);
    h = fma(h, e, h);
    r = fma(fma(-g, g, x), h, g);
    inv = 2.0 * fma(h, fma(-g, h, 0.5), h);
}

// Where the path through an edge's start vertex (along the edge) stops being the shorter one:
// the window (pseudo-source at (sx, sy) with s2 = |s|^2, sx measured from that vertex) beats it
// for x > x0 only, (x - sx)^2 + sy^2 < (x + a)^2 with a = the vertex's distance minus sigma.
// Rounded so that too little is cut, never too much (eps bounds that of 2 (a + sx), which nearly cancel
// where s lies near the edge's line beyond the vertex); beyond L: nothing of the window is left.
__device__ __forceinline__ float cut_at(float sx, float s2, float a, float L, float eps) {
    const float num = s2 - a * a - 2e-6f * (s2 + a * a) - eps * fabsf(sx), den = fmaf(2.0f, a + sx, eps);
    if (!(num > 0.0f)) return 0.0f;
    return den * L > num * 0.999f ? __fdividef(num, den) - 1e-5f * L : 2.0f * L;
}

// Evaluate a warp's queued tests (all lanes; lane k takes entry k < nev): the target's point in the
// frame of the entered half-edge, inside the cone or not, its length.  Paths that end with a
// straight piece from a vertex of the target's own face are kept apart from those that come
// through a window: a window wins over them unless they are shorter by more than the form's
// precision, so that a direction does not hang on the last bits of two equal lengths (FP32 form; in
// FP64 the shorter one is the one).  The lengths compared are the FP64 ones: FP32 lengths of their
// own cost two loads, a root and a record a target and 16 % of the kernel (16384 sources on a noisy
// sphere 2.86 against 2.45 ms).  One warp writes the direction of an improvement beside the
// length it lowered; a team's warps, which may lower one length at the same time, log them, and the
// log is read once the source is done.
template <class R, int PL, bool TEAM, bool LK>
__device__ __noinline__ void eval_tests(const cssi::GeoJob& J, const WaveLay& Y, unsigned char* b, unsigned char* e,
                                        GroupSm& sm, int nev, int lane, Links<LK> lk) {
    const DMesh& m = J.m;
    bool won = false, apart = false;
    int s = NONE;
    double d = 0.0;
    V2<R> t = vec2((R)0, (R)0);
    unsigned long long bits = 0;
    if (lane < nev) {
        const int4 w4 = at<int4>(e, Y.e[4])[lane];
        const int he = w4.x, j = w4.z;
        int vs = w4.y;
        const bool vertex = vs >= 0 && (vs & FROM_VERTEX);
        if (vertex) vs &= ~FROM_VERTEX;
        const double2 S = at<double2>(e, Y.e[0])[lane];
        const V2<R> rot = narrow<R>(at<double2>(e, Y.e[1])[lane]);
        const V2<R> d0 = narrow<R>(at<double2>(e, Y.e[2])[lane]), d1 = narrow<R>(at<double2>(e, Y.e[3])[lane]);
        const HeRec& r = m.he[he];
        const int k = he % 3;
        const double* bj = J.bary + 3 * (size_t)j;
        const double bv = bj[k == 2 ? 0 : k + 1], bc = bj[k == 0 ? 2 : k - 1];
        const double gx = bv * r.L + bc * r.cx - S.x, gy = bc * r.cy - S.y;
        const R fx = (R)gx, fy = (R)gy;
        const R qx = fx * rot.x + fy * rot.y, qy = fy * rot.x - fx * rot.y;
        // the cross products round with the distance, not with the edge
        const R tol = Rim<R>::t * (fabs(fx) + fabs(fy) + (R)r.L);
        const bool in = d0.x * qy - d0.y * qx <= tol * (fabs(d0.x) + fabs(d0.y)) &&
                        d1.x * qy - d1.y * qx >= -tol * (fabs(d1.x) + fabs(d1.y));
        const double n = sqrt(gx * gx + gy * gy), sig = vs < 0 ? 0.0 : at<double>(b, Y.vdist)[vs];
        d = sig + n;
        if (in && d < J.rc) {
            bool claimed;
            s = tab_insert(at<int32_t>(b, Y.tkey), Y.th_log, j, &sm.nt, Y.t_most, claimed);
            if (s < 0) atomicOr(&sm.err, css::ST_HASH_OVERFLOW);
            else {
                bits = (unsigned long long)__double_as_longlong(d);   // lengths start at infinity
                apart = sizeof(R) == 4 && vertex;
                won = atomicMin((unsigned long long*)at<double>(b, apart ? Y.tvert : Y.tdist) + s, bits) > bits;
            }
        }
        if (won) {
            if (vs < 0) {
                const R inv = n > 0.0 ? (R)1 / (R)n : (R)0;
                t = vec2(qx * inv, qy * inv);
            } else t = at<V2<R>>(b, Y.itan)[at<typename Index<PL>::type>(b, Y.vinfo)[vs]];
        }
    }
    if constexpr (TEAM) {
        if (won) {
            const int l = atomicAdd(&sm.nlog, 1);
            if (l >= Y.lg_cap) atomicOr(&sm.err, css::ST_HASH_OVERFLOW);
            else {
                at<double>(b, Y.ldist)[l] = d;
                at<V2<R>>(b, Y.ttan)[l] = t;
                at<int>(b, Y.lslot)[l] = apart ? s | FROM_VERTEX : s;
            }
        }
    } else {
        __syncwarp();
        // of the lanes that lowered one length only the lowest one's value is there now
        const int at_ = apart ? s + (1 << Y.th_log) : s;   // records of windows, then of vertices
        if (won && *((volatile unsigned long long*)at<double>(b, apart ? Y.tvert : Y.tdist) + s) == bits) {
            at<V2<R>>(b, Y.ttan)[at_] = t;
            if constexpr (LK) {
                const int4 w4 = at<int4>(e, Y.e[4])[lane];
                const double2 S = at<double2>(e, Y.e[0])[lane];
                const HeRec& r = m.he[w4.x];
                const int k = w4.x % 3;
                const double* bj = J.bary + 3 * (size_t)w4.z;
                const double bv = bj[k == 2 ? 0 : k + 1], bc = bj[k == 0 ? 2 : k - 1];
                link_back(m, w4.x, S, bv * r.L + bc * r.cx, bc * r.cy, 3, w4.y < 0 ? NONE : w4.y & ~FROM_VERTEX,
                          lk.p[(1 << Y.vh_log) + s]);
            }
        }
    }
}

// ------------------------------------------------------------------ one source
struct Win {
    double2 s, rot;     // the pseudo-source in the frame of half-edge he; image of its own frame's x axis
    double2 d0, d1;     // left and right rim of the cone, in its frame
    float b0, b1, key;
    int he, vs;
    int su, sv;         // slots of the edge's end vertices
};

template <class R, int PL, bool TEAM, bool LK>
struct Group {
    using Idx = typename Index<PL>::type;
    const cssi::GeoJob& J;
    const WaveLay& Y;
    unsigned char* b;      // tables
    unsigned char* h;      // ring
    unsigned char* e;      // this warp's queued tests and task list
    unsigned char* x;      // spill area
    GroupSm& sm;
    TeamSm* tm;
    int src, lane, wid, tid, T;
    float rcf;             // the cutoff, rounded up
    Links<LK> lk;
    int nev = 0;

    __device__ __forceinline__ void bar() const {
        if constexpr (TEAM) __syncthreads();
        else __syncwarp();
    }
    __device__ __forceinline__ int32_t* vkey() const { return at<int32_t>(b, Y.vkey); }
    __device__ __forceinline__ double* vdist() const { return at<double>(b, Y.vdist); }
    __device__ __forceinline__ Idx* vinfo() const { return at<Idx>(b, Y.vinfo); }
    __device__ __forceinline__ V2<R>* itan() const { return at<V2<R>>(b, Y.itan); }
    __device__ __forceinline__ float* iback() const { return at<float>(b, Y.iback); }
    __device__ __forceinline__ unsigned* ihc() const { return at<unsigned>(b, Y.ihc); }
    __device__ __forceinline__ Idx* waiting(int list) const { return at<Idx>(b, Y.emit) + list * Y.i_cap; }
    __device__ __forceinline__ int32_t* tkey() const { return at<int32_t>(b, Y.tkey); }
    __device__ __forceinline__ double* tdist() const { return at<double>(b, Y.tdist); }
    __device__ __forceinline__ double* tvert() const { return at<double>(b, Y.tvert); }

    __device__ __forceinline__ double dist_at(int s) const { return s < 0 ? CUDART_INF : *(volatile double*)(vdist() + s); }

    __device__ __forceinline__ void eval() {
        __syncwarp();
        if (nev) eval_tests<R, PL, TEAM, LK>(J, Y, b, e, sm, nev, lane, lk);
        __syncwarp();
        nev = 0;
    }

    // queue the particles of face bucket `key` for the lanes that have one; put(entry, particle)
    // writes an entry
    template <class Put>
    __device__ __forceinline__ void tests(bool has, int key, Put put) {
        int st = 0, cnt = 0;
        if (has) {
            st = J.fstart[key];
            cnt = J.fstart[key + 1] - st;
        }
#pragma unroll 1
        for (int r = 0; __any_sync(CSS_FULL, r < cnt); ++r) {
            int j = src;
            if (r < cnt) j = J.fitems[st + r];
            unsigned mk = __ballot_sync(CSS_FULL, j != src);
#pragma unroll 1
            while (mk) {   // as many as there is room for
                const int k = nev + __popc(mk & css::lanemask_lt());
                const bool now = j != src && (mk >> lane & 1u) && k < EV;
                if (now) put(k, j);
                const unsigned done = __ballot_sync(CSS_FULL, now);
                nev += __popc(done);
                mk &= ~done;
                if (TEAM ? nev == EV : __builtin_expect(nev == EV, 0)) eval();
            }
        }
    }
    __device__ __forceinline__ void put_test(int k, double2 s, double2 rot, double2 d0, double2 d1, int he, int vs, int j) {
        at<double2>(e, Y.e[0])[k] = s;
        at<double2>(e, Y.e[1])[k] = rot;
        at<double2>(e, Y.e[2])[k] = d0;
        at<double2>(e, Y.e[3])[k] = d1;
        at<int4>(e, Y.e[4])[k] = make_int4(he, vs, j, 0);
    }
    // every particle of the face is seen: a cone of no directions holds all
    __device__ __forceinline__ void put_open_test(int k, double2 s, double2 rot, int he, int vs, int j) {
        const double2 none = make_double2(0.0, 0.0);
        put_test(k, s, rot, none, none, he, vs, j);
    }

    // The interval of a ring entry: 16-bit fractions of the edge, rounded outward (0 and 1 are exact).
    static __device__ __forceinline__ int pack_interval(float b0, float b1, float L) {
        const float q = __fdividef(65535.0f, L);
        const int i0 = max(0, (int)floorf(b0 * q * 0.999999f - 0.01f));
        const int i1 = b1 >= L ? 65535 : min(65535, (int)ceilf(b1 * q * 1.000001f + 0.01f));
        return i0 | i1 << 16;
    }
    static __device__ __forceinline__ void unpack_interval(unsigned p, float L, float& b0, float& b1) {
        const unsigned i0 = p & 0xffffu, i1 = p >> 16;
        b0 = (float)i0 * (L * (1.0f / 65535.0f));
        b1 = i1 == 65535u ? L : (float)i1 * (L * (1.0f / 65535.0f));
    }

    __device__ __forceinline__ void store(unsigned char* to, const int* o, int k, const Win& w, int b01) {
        at<double2>(to, o[0])[k] = w.s;
        at<double2>(to, o[1])[k] = w.rot;
        at<double2>(to, o[2])[k] = w.d0;
        at<double2>(to, o[3])[k] = w.d1;
        at<int4>(to, o[4])[k] = make_int4(w.he, w.vs, __float_as_int(w.key), b01);
        at<typename Index<PL>::pair>(to, o[5])[k] = Index<PL>::make(w.su, w.sv);
    }
    // append windows (lanes with has): to the ring up to position `lim`, then to the spill area
    __device__ __forceinline__ void push(bool has, const Win& w, float L, int lim) {
        const unsigned mk = __ballot_sync(CSS_FULL, has);
        if (!mk) return;
        const int n = __popc(mk);
        int base = 0;
        if constexpr (TEAM) {
            if (lane == 0) base = atomicAdd(&sm.tail, n);
            base = __shfl_sync(CSS_FULL, base, 0);
        } else {
            base = sm.tail;
            __syncwarp();
            if (lane == 0) sm.tail = min(base + n, max(lim, base));
        }
        const int rank = __popc(mk & css::lanemask_lt());
        const int b01 = pack_interval(w.b0, w.b1, L);
        if (has && base + rank < lim) store(h, Y.r, (base + rank) & Y.r_mask, w, b01);
        if (TEAM ? base + n > lim : __builtin_expect(base + n > lim, 0)) {
            const int in = max(0, lim - base);   // those that went to the ring
            int sb = 0;
            if constexpr (TEAM) {
                if (lane == 0) sb = atomicAdd(&sm.stail, n - in);
                sb = __shfl_sync(CSS_FULL, sb, 0);
            } else {
                sb = sm.stail;
                __syncwarp();
                if (lane == 0) sm.stail = sb + n - in;
            }
            const int p = sb + rank - in;
            if (has && rank >= in) {
                if (p - sm.shead >= Y.s_cap) atomicOr(&sm.err, css::ST_WIN_OVERFLOW);
                else store(x, Y.s, p & (Y.s_cap - 1), w, b01);
            }
        }
        __syncwarp();
    }

    // a vertex distance less sigma
    __device__ __forceinline__ float rel(int slot, double sig) const {
        return slot < 0 ? 3e38f : f32(*(volatile double*)(vdist() + slot) - sig);
    }
    // cut [b0, b1] of an edge of length L by its end vertices' distances (less sigma) au, av; false if
    // nothing is left
    __device__ __forceinline__ bool cut(float sx, float sy, float au, float av, float L, float& b0, float& b1) const {
        const float sy2 = sy * sy, tx = L - sx, eps = 4.8e-7f * (fabsf(sx) + L);
        b0 = fmaxf(b0, cut_at(sx, sx * sx + sy2, au, L, eps));
        b1 = fminf(b1, L - cut_at(tx, tx * tx + sy2, av, L, eps));
        return b1 > b0;
    }
    // a lower bound on the lengths the window carries
    __device__ __forceinline__ float key_of(float sx, float sy, float sig, float b0, float b1) const {
        const float x = fminf(fmaxf(sx, b0), b1) - sx;
        return (sig + root(x * x + sy * sy)) * (1.0f - 3e-6f) - 4e-7f * (fabsf(sx) + b1);
    }

    // a vertex that got a smaller distance: its path's direction at the source and its last leg's
    // direction back; queued for starting windows if it is not queued yet
    // (angle `back` counter-clockwise from the first edge of corner hc; NaN where it is not known)
    __device__ __forceinline__ void improved(int slot, double d, V2<R> t, int hc, float back) {
        int i = vinfo()[slot];
        bool queued = false;
        if (i == (int)Index<PL>::none) {
            i = atomicAdd(&sm.ni, 1);
            if (TEAM ? i >= Y.i_cap : __builtin_expect(i >= Y.i_cap, 0)) {
                atomicOr(&sm.err, css::ST_HASH_OVERFLOW);
                return;
            }
            vinfo()[slot] = (Idx)i;
        } else queued = ihc()[i] & QUEUED;
        itan()[i] = t;
        iback()[i] = hc < 0 ? __int_as_float(0x7fffffff) : back;
        ihc()[i] = (hc < 0 ? 0u : (unsigned)hc) | QUEUED;
        atomicMin(&sm.emin, __float_as_uint(f32(d)));
        if (!queued) {   // a path record is in one of the lists at most once
            const int p = atomicAdd(&sm.nem[sm.cur], 1);
            if (p < Y.i_cap) waiting(sm.cur)[p] = (Idx)slot;
            else atomicOr(&sm.err, css::ST_HASH_OVERFLOW);
        }
    }
    __device__ __forceinline__ V2<R> tangent_of(int slot) const { return itan()[vinfo()[slot]]; }

    // slot of a vertex, entered with an infinite distance if it is new (distances are reset
    // when the source starts)
    __device__ __forceinline__ int vertex(int32_t v) {
        bool claimed;
        const int s = tab_insert(vkey(), Y.vh_log, v, &sm.nv, Y.v_most, claimed);
        if (s < 0) atomicOr(&sm.err, css::ST_HASH_OVERFLOW);
        return s;
    }

    __device__ __forceinline__ void seed(int f0, double b1, double b2);
    __device__ __forceinline__ void seed_at_vertex(int hc);
    __device__ __forceinline__ void emit(int ne, int lim, float kmin);
    __device__ __forceinline__ void wave(int head, int n);
    __device__ __forceinline__ void run(int item, int32_t* defer_list, int* defer_count, int* status,
                                        unsigned long long* counters);
};

// Start a source (warp 0): tests for its own face, distances of its corners, one window for
// each edge of its face.
template <class R, int PL, bool TEAM, bool LK>
__device__ __forceinline__ void Group<R, PL, TEAM, LK>::seed(int f0, double b1, double b2) {
    const DMesh& m = J.m;
    const bool c3 = lane < 3;
    const int hh = 3 * f0 + (c3 ? lane : 0);
    const HeRec r = m.he[hh];
    // the source from the corner's own weights (no cancellation next to a corner): (hx, hy) in the
    // frame of half-edge h, lx from its end; (ex, ey) the frame's x axis in the face's layout
    const int k0 = hh - 3 * f0;
    // (weights below zero by rounding are zero for all three lanes: a source that lies on an edge for one
    // and beside it for the others would see its corners in different directions)
    const double wt[3] = {fmax(1.0 - b1 - b2, 0.0), fmax(b1, 0.0), fmax(b2, 0.0)};
    const double wa = k0 == 0 ? wt[0] : (k0 == 1 ? wt[1] : wt[2]), wb = k0 == 0 ? wt[1] : (k0 == 1 ? wt[2] : wt[0]);
    const double wc = k0 == 0 ? wt[2] : (k0 == 1 ? wt[0] : wt[1]);
    const double hx = wb * r.L + wc * r.cx, lx = wa * r.L + wc * (r.L - r.cx), hy = wc * r.cy;
    double ax, ay, bx, by;
    unit_corner(m, f0, k0, ax, ay);
    unit_corner(m, f0, k0 + 1, bx, by);
    const double ex = (bx - ax) / r.L, ey = (by - ay) / r.L;
    const double vx = hy * ey - hx * ex, vy = -hy * ex - hx * ey;   // from the source to the corner, in the layout
    tests(lane == 0, m.frank ? m.frank[f0] : f0, [&](int k, int j) {   // half-edge 0's frame is the layout's
        put_open_test(k, make_double2(hx, hy), make_double2(1.0, 0.0), hh, NONE, j);
    });
    // a source on a corner (to the rounding of its position) has no direction to it: its windows start at the vertex, all around
    const double vd = sqrt(hx * hx + hy * hy);
    const unsigned on = __ballot_sync(CSS_FULL, c3 && vd <= 1e-15 * r.L);
    const int slot = c3 ? vertex(m.fv[hh]) : NONE;
    if (slot >= 0 && vd < J.rc && (on == 0 || (on >> lane & 1u))) {
        vdist()[slot] = vd;
        if constexpr (LK) lk.p[slot] = {NONE, 4 * f0 + k0, vd, make_double2(vd > 0.0 ? -vx / vd : 1.0, vd > 0.0 ? -vy / vd : 0.0)};
        if (!on && (m.htop[hh].x & css::EMITS))
            improved(slot, vd, vec2((R)(vx / vd), (R)(vy / vd)), vd > 1e-6 * r.L ? hh : NONE, atan2f((float)hy, (float)hx));
    }
    const int next = __shfl_sync(CSS_FULL, slot, lane == 2 ? 0 : lane + 1);
    __syncwarp();
    if (on) {
        seed_at_vertex(3 * f0 + __ffs(on) - 1);
        return;
    }
    const int tw = m.twin[hh];
    Win w;
    w.he = tw;
    w.vs = NONE;
    w.s = make_double2(lx, -hy);   // the twin runs from the edge's end to its start
    w.rot = make_double2(-ex, ey);
    w.d0 = make_double2(lx * ex + hy * ey, lx * ey - hy * ex);
    w.d1 = make_double2(vx, vy);
    w.b0 = 0.0f;
    w.b1 = (float)r.L;
    w.key = key_of((float)lx, (float)-hy, 0.0f, w.b0, w.b1);
    w.su = next;
    w.sv = slot;
    push(c3 && slot >= 0 && next >= 0 && tw >= 0 && w.key < rcf, w, w.b1, Y.r_mask + 1);
}

// A source on corner hc's vertex: one window opposite each corner of the vertex's ring, tests for
// the ring's faces, and the ring's vertices along its edges.  Directions come from unfolding
// the ring from the source's face, counter-clockwise for the first half and clockwise for the
// rest (at a vertex the direction in the source face's plane depends on that choice).  Serial:
// this is rare.
template <class R, int PL, bool TEAM, bool LK>
__device__ __forceinline__ void Group<R, PL, TEAM, LK>::seed_at_vertex(int hc) {
    const DMesh& m = J.m;
    const int32_t v = m.fv[hc];
    const int deg = m.ring_start[v + 1] - m.ring_start[v];
    const int f0 = hc / 3;
    double ax, ay, bx, by;
    unit_corner(m, f0, hc - 3 * f0, ax, ay);
    unit_corner(m, f0, hc - 3 * f0 + 1, bx, by);
    const double phi0 = atan2(by - ay, bx - ax);
    const int half = m.bnd[v] ? deg : (deg + 1) / 2;
    int left = deg;
#pragma unroll 1
    for (int dir = 0; dir < 2; ++dir) {
        int g = hc;
        double phi = phi0;   // direction of corner h's first edge in the source face's layout
#pragma unroll 1
        for (int q = 0; q < (dir == 0 ? half : deg) && left > 0; ++q) {
            if (q > 0 || dir == 1) {
                if (dir == 0) {   // the next corner, across this corner's last edge
                    const int f = g / 3, k = g - 3 * f;
                    const HeRec& a = m.he[g];
                    phi += atan2(a.cy, a.cx);
                    g = m.twin[3 * f + (k == 0 ? 2 : k - 1)];
                    if (g < 0) break;
                } else {          // the corner across this corner's first edge
                    const int o = m.twin[g];
                    if (o < 0) break;
                    const int fo = o / 3, kg = o - 3 * fo;
                    g = 3 * fo + (kg == 2 ? 0 : kg + 1);
                    const HeRec& a = m.he[g];
                    phi -= atan2(a.cy, a.cx);
                }
                if (g == hc) break;
            }
            --left;
            const int fh = g / 3, kh = g - 3 * fh;
            const HeRec r = m.he[g];
            const double co = cos(phi), si = sin(phi);
            tests(lane == 0 && g != hc, m.frank ? m.frank[fh] : fh, [&](int t, int j) {
                put_open_test(t, make_double2(0.0, 0.0), make_double2(co, -si), g, NONE, j);
            });
            const double ang = atan2(r.cy, r.cx), lc = sqrt(r.cx * r.cx + r.cy * r.cy);
            int slot = NONE;
            if (lane < 2) {   // the two other corners of the face, along its edges from the vertex
                const int hn = lane == 0 ? 3 * fh + (kh == 2 ? 0 : kh + 1) : 3 * fh + (kh == 0 ? 2 : kh - 1);
                const double d = lane == 0 ? r.L : lc, a = lane == 0 ? phi : phi + ang;
                slot = vertex(m.fv[hn]);
                if (slot >= 0 && d < J.rc) {
                    const unsigned long long bits = (unsigned long long)__double_as_longlong(d);
                    const unsigned long long old = atomicMin((unsigned long long*)(vdist() + slot), bits);
                    if (old > bits && (m.htop[hn].x & css::EMITS)) {
                        improved(slot, d, vec2((R)cos(a), (R)sin(a)), NONE, 0.0f);
                        if constexpr (LK) {   // along the edge, back to the source's corner
                            double px, py, sx, sy;
                            unit_corner(m, fh, hn - 3 * fh, px, py);
                            unit_corner(m, fh, kh, sx, sy);
                            lk.p[slot] = {NONE, 4 * fh + (hn - 3 * fh), d, make_double2((sx - px) / d, (sy - py) / d)};
                        }
                    }
                }
            }
            const int s1 = __shfl_sync(CSS_FULL, slot, 0), s2 = __shfl_sync(CSS_FULL, slot, 1);
            __syncwarp();
            const int hop = 3 * fh + (kh == 2 ? 0 : kh + 1);
            Win w;
            w.he = m.twin[hop];
            w.vs = NONE;
            const HeRec o = m.he[hop];
            w.s = make_double2(o.L - o.cx, -o.cy);
            // the twin's x axis runs from the face's far corner c to the first edge's end
            const double tx = (r.L - r.cx) / o.L, ty = -r.cy / o.L;
            w.rot = make_double2(tx * co - ty * si, -(tx * si + ty * co));
            w.d0 = make_double2(r.cx * co - r.cy * si, r.cx * si + r.cy * co);
            w.d1 = make_double2(r.L * co, r.L * si);
            w.b0 = 0.0f;
            w.b1 = (float)o.L;
            w.key = key_of((float)w.s.x, (float)w.s.y, 0.0f, w.b0, w.b1);
            w.su = s2;
            w.sv = s1;
            push(lane == 0 && s1 >= 0 && s2 >= 0 && w.he >= 0 && w.key < rcf, w, w.b1, Y.r_mask + 1);
            __syncwarp();
        }
    }
}

// Vertices whose distance is final (at most kmin, the smallest key that waits) start a window on
// the edge opposite each corner of their ring that a shortest path through them can enter; the
// particles of those faces are tested as well (a path may end right behind the vertex).
// A shortest path through an interior vertex of angle sum T leaves it at least pi away from its
// incoming direction on both sides, so within [b + pi, b + T - pi] of the direction b back along
// any shortest path to it.  The window is clipped to that range, widened by SHADOW_TOL for the
// rounding of b and the corner angles.  Vertices without a known b, boundary and non-manifold
// ones start windows over their whole ring.
template <class R, int PL, bool TEAM, bool LK>
__device__ __forceinline__ void Group<R, PL, TEAM, LK>::emit(int ne, int lim, float kmin) {
    const DMesh& m = J.m;
    const int from = sm.cur, to = 1 - from;
    bar();
    if (tid == 0) {
        sm.nem[to] = 0;
        sm.cur = to;
        sm.emin = 0x7f800000u;
    }
    bar();
#pragma unroll 1
    for (int base = tid - lane; base < ne; base += T) {
        const int it = base + lane;
        int vs = 0;
        bool go = false;
        double dv = 0.0;
        if (it < ne) {
            vs = waiting(from)[it];
            dv = vdist()[vs];
            go = dv <= (double)kmin;
            if (!go) {
                waiting(to)[atomicAdd(&sm.nem[to], 1)] = (Idx)vs;
                atomicMin(&sm.emin, __float_as_uint(__double2float_rd(dv)));
            }
        }
        int rs = 0, len = 0;
        float lo = -INFINITY, hi = INFINITY, th = 0.0f;
        if (go) {
            const int i = vinfo()[vs];
            const unsigned hb = ihc()[i] & ~QUEUED;
            const float bk = iback()[i] + m.cang[hb].x;   // NaN where either is not known
            ihc()[i] = hb;
            const int vid = vkey()[vs];
            rs = m.ring_start[vid];
            len = m.ring_start[vid + 1] - rs;
            if (bk == bk) {
                th = (float)m.theta[vid];
                lo = bk + 3.14159265f - geo::SHADOW_TOL;
                lo -= th * floorf(__fdividef(lo, th));
                hi = lo + (th - 6.28318531f + 2.0f * geo::SHADOW_TOL);
            }
        }
        // one lane per (vertex, corner)
        const int incl = geo::warp_incl_scan(len, lane);
        const int total = __shfl_sync(CSS_FULL, incl, 31);
#pragma unroll 1
        for (int tb = 0; tb < total; tb += 32) {
            const int t = tb + lane;
            const int owner = geo::scan_owner(incl, t);
            const int o_rs = __shfl_sync(CSS_FULL, rs, owner), o_ex = __shfl_sync(CSS_FULL, incl - len, owner);
            const int o_vs = __shfl_sync(CSS_FULL, vs, owner);
            const double o_dv = __shfl_sync(CSS_FULL, dv, owner);
            const float o_lo = __shfl_sync(CSS_FULL, lo, owner), o_hi = __shfl_sync(CSS_FULL, hi, owner);
            const float o_th = __shfl_sync(CSS_FULL, th, owner);
            bool hit = false;
            int hc = 0, f = 0;
            float c0 = 0.0f, c1 = 0.0f, wid_c = 0.0f;   // the lit part of the corner, from its first edge
            if (t < total) {
                hc = m.ring[o_rs + (t - o_ex)];
                f = hc / 3;
                if (o_th == 0.0f) hit = true;
                else {
                    const float2 cw = m.cang[hc];
                    wid_c = cw.y;
                    c0 = INFINITY;
                    c1 = -INFINITY;
#pragma unroll 1
                    for (int s = -1; s <= 1; ++s) {   // one turn either way
                        const float a = cw.x + (float)s * o_th;
                        const float l = fmaxf(a, o_lo), r = fminf(a + cw.y, o_hi);
                        if (!(r < l)) {
                            hit = true;
                            c0 = fminf(c0, l - a);
                            c1 = fmaxf(c1, r - a);
                        }
                    }
                }
            }
            tests(hit, hit ? m.htop[hc].w : 0, [&](int k, int j) {
                put_open_test(k, make_double2(0.0, 0.0), make_double2(1.0, 0.0), hc, o_vs | FROM_VERTEX, j);
            });
            Win w;
            bool ok = false;
            float L = 0.0f;
            if (hit) {
                const int k = hc - 3 * f, hop = 3 * f + (k == 2 ? 0 : k + 1);
                w.he = m.twin[hop];
                if (w.he >= 0) {
                    const HeRec r = m.he[hop];
                    L = (float)r.L;
                    w.vs = o_vs | FIRST;
                    w.s = make_double2(r.L - r.cx, -r.cy);
                    w.rot = make_double2(1.0, 0.0);
                    w.b0 = 0.0f;
                    w.b1 = L;
                    if (o_th != 0.0f) {
                        // where the directions c0 and c1 meet the opposite edge, as a part of it
                        const css::HeRec32 q = m.he32[hc];
                        const float ex = q.cx - q.L, ey = q.cy;
                        if (c0 > 1e-5f) {
                            const float s = __sinf(c0), c = __cosf(c0);
                            const float x = fminf(fmaxf(__fdividef(q.L * s, ey * c - ex * s), 0.0f), 1.0f);
                            w.b1 = fminf(L, L * (1.0f - x) + 1e-5f * L);
                        }
                        if (c1 < wid_c - 1e-5f) {
                            const float s = __sinf(c1), c = __cosf(c1);
                            const float x = fminf(fmaxf(__fdividef(q.L * s, ey * c - ex * s), 0.0f), 1.0f);
                            w.b0 = fmaxf(0.0f, L * (1.0f - x) - 1e-5f * L);
                        }
                    }
                    w.d0 = make_double2((double)w.b0 - w.s.x, -w.s.y);
                    w.d1 = make_double2((w.b1 == L ? r.L : (double)w.b1) - w.s.x, -w.s.y);
                    const int4 tp = m.htop[w.he];
                    w.su = vertex(tp.x & css::VMASK);
                    w.sv = vertex(tp.y & css::VMASK);
                    const float fx = f32(w.s.x), fy = f32(w.s.y);
                    ok = cut(fx, fy, rel(w.su, o_dv), rel(w.sv, o_dv), L, w.b0, w.b1) && w.su >= 0 && w.sv >= 0;
                    w.key = key_of(fx, fy, f32(o_dv), w.b0, w.b1);
                    ok = ok && w.key < rcf;
                }
            }
            push(ok, w, L, lim);
        }
    }
}

// Unfold the windows head .. head + n of the ring (at most one per thread).
template <class R, int PL, bool TEAM, bool LK>
__device__ __forceinline__ void Group<R, PL, TEAM, LK>::wave(int head, int n) {
    const DMesh& m = J.m;
    const bool on = tid < n;
    const int s = (head + tid) & Y.r_mask;
    const int4 w4 = on ? at<int4>(h, Y.r[4])[s] : make_int4(0, NONE, 0, 0);
    const int he = w4.x;
    const bool first = w4.y >= 0 && (w4.y & FIRST);
    const int vs = w4.y < 0 ? NONE : w4.y & ~FIRST;
    const int4 tp = m.htop[he];
    const HeRec r = m.he[he];
    const css::HeRec32 q = m.he32[he];
    tests(on, tp.w, [&](int k, int j) {
        put_test(k, at<double2>(h, Y.r[0])[s], at<double2>(h, Y.r[1])[s], at<double2>(h, Y.r[2])[s], at<double2>(h, Y.r[3])[s],
                 he, vs, j);
    });
    const double2 S = at<double2>(h, Y.r[0])[s];
    const typename Index<PL>::pair ends = at<typename Index<PL>::pair>(h, Y.r[5])[s];
    const int su = on ? (int)ends.x : NONE, sv = on ? (int)ends.y : NONE;
    float b0, b1;
    unpack_interval((unsigned)w4.w, q.L, b0, b1);
    const double sig = vs < 0 ? 0.0 : vdist()[vs];
    const float fsx = f32(S.x), fsy = f32(S.y), fsig = f32(sig);
    const bool act = on && cut(fsx, fsy, rel(su, sig), rel(sv, sig), q.L, b0, b1) && key_of(fsx, fsy, fsig, b0, b1) < rcf;
    // the far corner seen from s, in FP32 (fgx, fgy), and its side of the cone's rims
    const float fgx = q.cx - fsx, fgy = q.cy - fsy, size = fabsf(fsx) + fabsf(fsy) + q.L;
    const float em = 4e-6f * size;   // bounds the rounding of FP32 crossings
    const float xc = fsx - fgx * __fdividef(fsy, fgy);
    bool in0, in1, beyond0, beyond1;   // c on or right of the left rim, on or left of the right rim; strictly
    {
        const double2 rot = at<double2>(h, Y.r[1])[s], d0 = at<double2>(h, Y.r[2])[s], d1 = at<double2>(h, Y.r[3])[s];
        const float rx = f32(rot.x), ry = f32(rot.y), px = fgx * rx + fgy * ry, py = fgy * rx - fgx * ry;
        const float ax = f32(d0.x), ay = f32(d0.y), bx = f32(d1.x), by = f32(d1.y);
        const float cr0 = ax * py - ay * px, cr1 = bx * py - by * px;   // < 0: c lies right of the rim
        const float t = 8e-6f * (fabsf(fgx) + fabsf(fgy) + size);
        const float t0 = t * (fabsf(ax) + fabsf(ay)), t1 = t * (fabsf(bx) + fabsf(by));
        in0 = cr0 <= t0;
        beyond0 = cr0 < -t0;
        in1 = cr1 >= -t1;
        beyond1 = cr1 > t1;
        const bool near = on && ((in0 && !beyond0) || (in1 && !beyond1));
        if (TEAM ? near : __builtin_expect(near, 0)) {   // too close to a rim for FP32
            const double gx = r.cx - S.x, gy = r.cy - S.y;
            const double ex = gx * rot.x + gy * rot.y, ey = gy * rot.x - gx * rot.y;
            const double tg = RIM_MIN * (fabs(gx) + fabs(gy));
            const double e0 = tg * (fabs(d0.x) + fabs(d0.y)), e1 = tg * (fabs(d1.x) + fabs(d1.y));
            const double c0 = d0.x * ey - d0.y * ex, c1 = d1.x * ey - d1.y * ex;
            in0 = c0 <= e0;
            beyond0 = c0 < -e0;
            in1 = c1 >= -e1;
            beyond1 = c1 > e1;
        }
    }
    const bool left = act && beyond0 && xc > b0 - em && r.tl >= 0, right = act && beyond1 && xc < b1 + em && r.tr >= 0;
    const bool cin = act && in0 && in1 && xc >= b0 - em && xc <= b1 + em;
    // distance candidates: the far corner, and the two ends of a window that just started
    int sc = NONE;
    const int nq = (TEAM ? __syncthreads_or(first) : __any_sync(CSS_FULL, first)) ? 3 : 1;
#pragma unroll 1
    for (int a = 0; a < nq; ++a) {
        const bool has = a == 0 ? cin : (first && act && (a == 1 ? b0 <= 0.0f : b1 >= q.L));
        const float fvx = a == 0 ? fgx : (a == 1 ? -fsx : q.L - fsx), fvy = a == 0 ? fgy : -fsy;
        const int vtop = a == 0 ? tp.z : (a == 1 ? tp.x : tp.y);
        const float fd = fsig + root(fvx * fvx + fvy * fvy), fe = 1e-6f * (fd + size);   // its rounding
        int slot = a == 1 ? su : sv;
        if (a == 0) {
            slot = left || right || cin ? vertex(vtop & css::VMASK) : NONE;
            sc = slot;
            bar();
        }
        unsigned long long bits = 0, old = 0;
        double d = 0.0;
        V2<R> t = vec2((R)0, (R)0);
        if (has && slot >= 0 && fd - fe < rcf && fd - fe < f32(dist_at(slot)) * (1.0f + 3e-7f)) {
            // the other vertices' distances only cut windows: an FP32 upper bound will do
            if (vtop & css::EMITS) {
                const double vx = a == 0 ? r.cx - S.x : (a == 1 ? -S.x : r.L - S.x), vy = a == 0 ? r.cy - S.y : -S.y;
                double n, inv;
                roots(vx * vx + vy * vy, n, inv);
                d = sig + n;
                if (vs < 0) {
                    const V2<R> rot = narrow<R>(at<double2>(h, Y.r[1])[s]);
                    const R gx = (R)vx, gy = (R)vy, ri = (R)inv;
                    t = vec2((gx * rot.x + gy * rot.y) * ri, (gy * rot.x - gx * rot.y) * ri);
                }
            } else d = f64(fd + fe);
            bits = (unsigned long long)__double_as_longlong(d);
            if (d < J.rc) old = atomicMin((unsigned long long*)(vdist() + slot), bits);
        }
        bar();
        if (old > bits && (vtop & css::EMITS) && *(volatile unsigned long long*)(vdist() + slot) == bits) {
            if (vs >= 0) t = tangent_of(vs);
            const int f = he / 3, k = he - 3 * f;
            const int hc = a == 0 ? 3 * f + (k == 0 ? 2 : k - 1) : (a == 1 ? he : m.twin[he]);
            // the last leg back, from the corner's first edge: c -> u, u -> v, v -> u
            const float ex = a == 0 ? -q.cx : (a == 1 ? 1.0f : -1.0f), ey = a == 0 ? -q.cy : 0.0f;
            improved(slot, d, t, fvx * fvx + fvy * fvy > 1e-6f * size * size ? hc : NONE,
                     atan2f(ey * fvx - ex * fvy, -ex * fvx - ey * fvy));
            if constexpr (LK)
                link_back(m, he, S, a == 0 ? r.cx : (a == 1 ? 0.0 : r.L), a == 0 ? r.cy : 0.0, a == 0 ? 2 : a - 1, vs,
                          lk.p[slot]);
        }
        bar();
    }
    // The children, side 0 across the edge u -> c, side 1 across c -> v: one lane each, packed densely
    // (a window has one child on average, at most two).  A child's lane reads its parent's
    // window from the ring again; the parent's slots are free once the last round has read them.
    // (the corner bounds a child's cone only where it splits it: a rim that moved to every corner within
    // its tolerance would leave a gap of several tolerances after a chain of them, and the sliver between
    // has no windows of its own behind flat vertices)
    const unsigned lm = __ballot_sync(CSS_FULL, left), rm = __ballot_sync(CSS_FULL, right);
    const int nleft = __popc(lm), total = nleft + __popc(rm);
    unsigned char* task = e + Y.e_task;
    if (left) task[__popc(lm & css::lanemask_lt())] = (unsigned char)(lane | (beyond1 ? 64 : 0));
    if (right) task[nleft + __popc(rm & css::lanemask_lt())] = (unsigned char)(lane | 32 | (beyond0 ? 64 : 0));
    __syncwarp();
#pragma unroll 1
    for (int base = 0; base < total; base += 32) {
        const bool is = base + lane < total;
        const int code = is ? task[base + lane] : 0;
        const int par = code & 31;
        const float pb0 = __shfl_sync(CSS_FULL, b0, par), pb1 = __shfl_sync(CSS_FULL, b1, par);
        const int psu = __shfl_sync(CSS_FULL, su, par), psv = __shfl_sync(CSS_FULL, sv, par);
        const int psc = __shfl_sync(CSS_FULL, sc, par);
        const int ps = (head + tid - lane + par) & Y.r_mask;
        const int4 pw = at<int4>(h, Y.r[4])[ps];
        const double2 PS = at<double2>(h, Y.r[0])[ps];
        const double2 rot = at<double2>(h, Y.r[1])[ps];
        Win w;
        w.d0 = at<double2>(h, Y.r[2])[ps];
        w.d1 = at<double2>(h, Y.r[3])[ps];
        __syncwarp();
        bool has = is;
        float Lc = 1.0f;
        if (is) {
            const bool a = code & 32;
            const HeRec pr = m.he[pw.x];
            const css::HeRec32 pq = m.he32[pw.x];
            w.he = a ? pr.tr : pr.tl;
            w.vs = pw.y < 0 ? NONE : pw.y & ~FIRST;
            const double psig = w.vs < 0 ? 0.0 : vdist()[w.vs];
            const double cx = pr.cx - PS.x, cy = pr.cy - PS.y;
            w.su = a ? psc : psu;
            w.sv = a ? psv : psc;
            if (code & 64) {
                const double2 pc = make_double2(cx * rot.x + cy * rot.y, cy * rot.x - cx * rot.y);
                if (a) w.d0 = pc;
                else w.d1 = pc;
            }
            const double co = a ? pr.cr : pr.cl, si = a ? pr.sr : pr.sl;
            const double ux = a ? -cx : PS.x, uy = a ? -cy : PS.y;   // s from the child edge's start
            w.s = make_double2(ux * co + uy * si, uy * co - ux * si);
            if (__double2hiint(w.s.y) >= 0) w.s.y = 0.0;   // rounding: s never lies above the edge
            w.rot = make_double2(rot.x * co + rot.y * si, rot.y * co - rot.x * si);
            // the interval: where the rays through b0 and b1 meet the child's edge, rounded outward
            const float sx = f32(PS.x), sy = f32(PS.y), sg = f32(psig);
            const float pem = 4e-6f * (fabsf(sx) + fabsf(sy) + pq.L);
            const float pxc = sx - (pq.cx - sx) * __fdividef(sy, pq.cy - sy);
            const float ax = a ? pq.cx : 0.0f, ay = a ? pq.cy : 0.0f;
            const float ex = a ? pq.L - pq.cx : pq.cx, ey = a ? -pq.cy : pq.cy;
            Lc = root(ex * ex + ey * ey);
            const float vx = sx - ax, vy = sy - ay;
            const float x0 = pb0 - sx, x1 = pb1 - sx;   // ray directions (x, -sy)
            const float m0 = -vx * sy - vy * x0, e0 = -ex * sy - ey * x0;
            const float m1 = -vx * sy - vy * x1, e1 = -ex * sy - ey * x1;
            // rounding of a crossing: that of the coordinates (em), and that of the ray's direction, which
            // grows as s nears the point the ray goes through
            const float emc = pem + 4e-6f * Lc, emd = pem * (Lc + pq.L);
            const float p0 = emc + __fdividef(emd, fmaxf(fabsf(x0), -sy)), p1 = emc + __fdividef(emd, fmaxf(fabsf(x1), -sy));
            w.b0 = a && pxc >= pb0 ? 0.0f : fmaxf(0.0f, fminf(e0 != 0.0f ? __fdividef(m0, e0) : 0.0f, 1.0f) * Lc - p0);
            w.b1 = !a && pxc <= pb1 ? Lc : fminf(Lc, fmaxf(e1 != 0.0f ? __fdividef(m1, e1) : 0.0f, 0.0f) * Lc + p1);
            const float fx = f32(w.s.x), fy = f32(w.s.y);
            has = cut(fx, fy, rel(w.su, psig), rel(w.sv, psig), Lc, w.b0, w.b1) && psc >= 0;
            w.key = key_of(fx, fy, sg, w.b0, w.b1);
            has = has && w.key < rcf;
        }
        push(has, w, Lc, head + Y.r_mask + 1 + (!TEAM && base + 32 >= total ? n : 0));
    }
}

template <class R, int PL, bool TEAM, bool LK>
__device__ __forceinline__ void Group<R, PL, TEAM, LK>::run(int item, int32_t* defer_list, int* defer_count, int* status,
                                                        unsigned long long* counters) {
    const DMesh& m = J.m;
    const int f0 = J.face[src];
    const double* bs = J.bary + 3 * (size_t)src;
    // empty tables; distances start at infinity
    {
        const int4 none = make_int4(-1, -1, -1, -1), inf = make_int4(0, 0x7ff00000, 0, 0x7ff00000);
#pragma unroll 1
        for (int k = tid; k < (1 << Y.vh_log) / 4; k += T) at<int4>(b, Y.vkey)[k] = none;
#pragma unroll 1
        for (int k = tid; k < (1 << Y.vh_log) / 2; k += T) at<int4>(b, Y.vdist)[k] = inf;
#pragma unroll 1
        for (int k = tid; k < (int)sizeof(Idx) * (1 << Y.vh_log) / 16; k += T) at<int4>(b, Y.vinfo)[k] = none;
#pragma unroll 1
        for (int k = tid; k < (1 << Y.th_log) / 4; k += T) at<int4>(b, Y.tkey)[k] = none;
#pragma unroll 1
        for (int k = tid; k < (1 << Y.th_log) / 2; k += T) {
            at<int4>(b, Y.tdist)[k] = inf;
            if (sizeof(R) == 4) at<int4>(b, Y.tvert)[k] = inf;
        }
    }
    if (tid == 0) {
        sm.head = sm.tail = sm.shead = sm.stail = sm.nem[0] = sm.nem[1] = sm.cur = 0;
        sm.nv = sm.ni = sm.nt = sm.nlog = sm.err = 0;
        sm.emin = 0x7f800000u;
    }
    bar();
    if (wid == 0) seed(f0, bs[1], bs[2]);
    unsigned nprop = 0;
    int waves = 0, lim = Y.r_mask + 1;
    for (;;) {
        bar();
        const int head = sm.head, ne = sm.nem[sm.cur], waits = sm.stail - sm.shead;
        int tail = min(sm.tail, lim), err = sm.err;   // a team's claims may run past the ring's end
        if (++waves > Y.max_waves) err |= css::ST_ITER_LIMIT;
        bar();
        const bool done = err || (head == tail && ne == 0 && waits == 0);
        if (TEAM ? done : __builtin_expect(done, 0)) {
            if (tid == 0) sm.err = err;
            break;
        }
        // spilled windows come back as the ring empties
        const int back = waits > 0 && tail - head < T ? min(waits, Y.r_mask + 1 - (tail - head)) : 0;
        if (TEAM ? back > 0 : __builtin_expect(back > 0, 0)) {
            const int from = sm.shead;
#pragma unroll 1
            for (int k = tid; k < back; k += T) {
                const int i = (from + k) & (Y.s_cap - 1), o = (tail + k) & Y.r_mask;
                at<double2>(h, Y.r[0])[o] = at<double2>(x, Y.s[0])[i];
                at<double2>(h, Y.r[1])[o] = at<double2>(x, Y.s[1])[i];
                at<double2>(h, Y.r[2])[o] = at<double2>(x, Y.s[2])[i];
                at<double2>(h, Y.r[3])[o] = at<double2>(x, Y.s[3])[i];
                at<int4>(h, Y.r[4])[o] = at<int4>(x, Y.s[4])[i];
                at<typename Index<PL>::pair>(h, Y.r[5])[o] = at<typename Index<PL>::pair>(x, Y.s[5])[i];
            }
            tail += back;
            bar();
            if (tid == 0) sm.shead = from + back;
        }
        if (tid == 0) sm.tail = tail;
        lim = head + Y.r_mask + 1;
        bar();
        if (ne > 0) {
            float km = INFINITY;
#pragma unroll 1
            for (int k = head + tid; k < tail; k += T) km = fminf(km, __int_as_float(at<int4>(h, Y.r[4])[k & Y.r_mask].z));
#pragma unroll 1
            for (int k = sm.shead + tid; k < sm.stail; k += T)
                km = fminf(km, __int_as_float(at<int4>(x, Y.s[4])[k & (Y.s_cap - 1)].z));
            km = __uint_as_float(__reduce_min_sync(CSS_FULL, __float_as_uint(km)));
            if constexpr (TEAM) {
                if (lane == 0) tm->km[wid] = km;
                __syncthreads();
                for (int w = 0; w < (T >> 5); ++w) km = fminf(km, tm->km[w]);
            }
            if (head == tail || __uint_as_float(sm.emin) <= km) {
                emit(ne, lim, km);
                bar();
                tail = min(sm.tail, lim);
            }
        }
        const int n = min(tail - head, T);
        wave(head, n);
        nprop += n;
        if (!TEAM) lim += n;   // the popped slots were free for the last children
        bar();
        if (tid == 0) {
            sm.head = head + n;
            if (TEAM) sm.tail = min(sm.tail, lim);
        }
    }
    eval();
    bar();
    const int err = sm.err;
    if (err) {   // a patch too large for this pass: the second pass takes the source, or the host hears of it
        if (tid == 0) {
            if (defer_list) {
                defer_list[atomicAdd(defer_count, 1)] = item;
                atomicAdd(counters + 4, 1ull);
            } else atomicOr(status, err);
        }
        return;
    }
    // the targets in particle order (every sum below runs in that order, so it does not depend on
    // the order of discovery)
    const int nt = sm.nt;
    int* list = at<int>(b, Y.tlist);
    int* ord = list + (1 << Y.th_log);
    if (tid == 0) sm.head = 0;
    bar();
#pragma unroll 1
    for (int k = tid; k < (1 << Y.th_log); k += T)
        if (tkey()[k] != NONE) list[atomicAdd(&sm.head, 1)] = k;
    bar();
    if (nt <= 128) {
#pragma unroll 1
        for (int k = tid; k < nt; k += T) {
            const int s = list[k], j = tkey()[s];
            int rank = 0;
#pragma unroll 1
            for (int q = 0; q < nt; ++q) rank += tkey()[list[q]] < j;
            ord[rank] = s;
        }
    } else {   // bitonic sort
        int n2 = 128;
        while (n2 < nt) n2 <<= 1;
#pragma unroll 1
        for (int k = tid; k < n2; k += T) ord[k] = k < nt ? list[k] : NONE;
        bar();
#pragma unroll 1
        for (int size = 2; size <= n2; size <<= 1)
#pragma unroll 1
            for (int step = size >> 1; step > 0; step >>= 1) {
#pragma unroll 1
                for (int k = tid; k < n2 / 2; k += T) {
                    const int lo = 2 * k - (k & (step - 1)), hi = lo + step;
                    const int a = ord[lo], c = ord[hi];
                    const int ka = a < 0 ? INT_MAX : tkey()[a], kc = c < 0 ? INT_MAX : tkey()[c];
                    if ((ka > kc) == !(lo & size)) { ord[lo] = c; ord[hi] = a; }
                }
                bar();
            }
    }
    bar();
    // a team: the log entries that hold each target's distance (through a window, and from a vertex)
    int* own = list;
    int* ownv = ord + (1 << Y.th_log);
    if constexpr (TEAM) {
        for (int l = tid; l < min(sm.nlog, Y.lg_cap); l += T) {
            const int c = at<int>(b, Y.lslot)[l], s = c & ~FROM_VERTEX;
            const bool vertex = sizeof(R) == 4 && (c & FROM_VERTEX);
            if (at<double>(b, Y.ldist)[l] == (vertex ? tvert() : tdist())[s]) (vertex ? ownv : own)[s] = l;
        }
        bar();
    }
    double fx = 0.0, fy = 0.0, en = 0.0;
    const double* fr = m.frame + 9 * (size_t)f0;
#pragma unroll 1
    for (int k = tid; k < nt; k += T) {
        const int s = ord[k];
        int l = TEAM ? own[s] : s;
        double d = tdist()[s];   // in units of the mesh until the form's choice is made
        if constexpr (sizeof(R) == 4) {
            const double dv = tvert()[s];
            const int lv = TEAM ? ownv[s] : s + (1 << Y.th_log);
            if (dv < d - TIE32 * dv) {
                l = lv;
                d = dv;
            }
        }
        d *= m.unit;
        const V2<R> t = at<V2<R>>(b, Y.ttan)[l];
        const double tx = (double)t.x, ty = (double)t.y;
        if (J.want_pairs && k < J.pair_cap) {
            const size_t o = (size_t)src * J.pair_cap + k;
            J.pj[o] = tkey()[s];
            J.pd[o] = d;
            J.pt[3 * o] = tx * fr[3] + ty * fr[6];
            J.pt[3 * o + 1] = tx * fr[4] + ty * fr[7];
            J.pt[3 * o + 2] = tx * fr[5] + ty * fr[8];
        }
        if constexpr (LK) {   // the pair's legs, from the target back to the source
            if (k < J.pair_cap) {
                const size_t o = (size_t)item * J.pair_cap + k;
                Link l = lk.p[(1 << Y.vh_log) + s];
                int nl = 0;
                for (;;) {
                    if (nl >= J.lmax) { nl = -1; break; }
                    const size_t a = o * J.lmax + nl;
                    J.lfk[a] = l.fk;
                    J.ldir[2 * a] = l.dir.x;
                    J.ldir[2 * a + 1] = l.dir.y;
                    J.llen[a] = l.len * m.unit;
                    ++nl;
                    if (l.par < 0) break;
                    l = lk.p[l.par];
                }
                J.lnum[o] = nl;
            }
        }
        if (J.want_forces) {
            const double du = geo::pot_dudl(J.pot, d);
            fx += du * tx;
            fy += du * ty;
            en += 0.5 * geo::pot_u(J.pot, d);
        }
    }
    fx = css::warp_sum(fx);
    fy = css::warp_sum(fy);
    en = css::warp_sum(en);
    if constexpr (TEAM) {
        if (lane == 0) {
            tm->fx[wid] = fx;
            tm->fy[wid] = fy;
            tm->en[wid] = en;
        }
        __syncthreads();
        if (tid == 0)
            for (int w = 1; w < (T >> 5); ++w) {
                fx += tm->fx[w];
                fy += tm->fy[w];
                en += tm->en[w];
            }
    }
    if (tid == 0) {
        if (J.want_forces) {
            J.force[3 * (size_t)src] = fx * fr[3] + fy * fr[6];
            J.force[3 * (size_t)src + 1] = fx * fr[4] + fy * fr[7];
            J.force[3 * (size_t)src + 2] = fx * fr[5] + fy * fr[8];
            if (J.epot) atomicAdd(J.epot, en);
        }
        if (J.pcnt) J.pcnt[src] = nt;
        if (J.want_pairs && nt > J.pair_cap) atomicOr(status, css::ST_PAIR_OVERFLOW);
        atomicAdd(counters + 0, 1ull);
        atomicAdd(counters + 1, (unsigned long long)nprop);
        atomicAdd(counters + 2, (unsigned long long)nprop);
        atomicAdd(counters + 3, (unsigned long long)nt);
    }
}

// PL 1: tables and ring in shared memory, 0: in the group's slice of global memory.  TEAM: the
// warps of a CTA work on one source, else each warp on its own.  Persistent: groups pull work
// items from a counter.
template <class R, int PL, bool TEAM, bool LK>
__global__ void __launch_bounds__(256, LK ? 1 : 2) k_waves(const __grid_constant__ cssi::GeoJob job0, const cssi::GeoJob* jobs,
                                                  const __grid_constant__ cssi::GeoQueue q,
                                                  const __grid_constant__ WaveWs g, int* work, int* status,
                                                  unsigned long long* counters) {
    __shared__ GroupSm sms[TEAM ? 1 : MAXW];
    TeamSm* tm = nullptr;
    if constexpr (TEAM) {
        __shared__ TeamSm team;
        tm = &team;
    }
    extern __shared__ __align__(16) unsigned char dsm[];
    const int wpc = blockDim.x >> 5, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int in_cta = TEAM ? 0 : wid, groups = TEAM ? 1 : wpc;
    GroupSm& sm = sms[in_cta];
    const int gid = blockIdx.x * groups + in_cta;
    // each group's ring and (PL 1) tables, then each warp's queued tests
    unsigned char* h = dsm + (size_t)in_cta * (g.lay.h_bytes + (PL == 1 ? g.lay.t_bytes : 0));
    unsigned char* b = PL == 1 ? h + g.lay.h_bytes : (unsigned char*)g.base + (size_t)gid * g.stride;
    unsigned char* x = (unsigned char*)g.base + (size_t)gid * g.stride + (PL == 1 ? 0 : g.lay.t_bytes);
    unsigned char* e = dsm + (size_t)groups * (g.lay.h_bytes + (PL == 1 ? g.lay.t_bytes : 0)) + (size_t)wid * g.lay.e_bytes;
    const int nitems = q.item_count ? min(*(volatile const int*)q.item_count, q.nitems) : q.nitems;
    const int tile = TEAM ? 1 : max(1, q.tile);
    for (;;) {
        int first = 0;
        if constexpr (TEAM) {
            __syncthreads();
            if (threadIdx.x == 0) sm.item = atomicAdd(work, 1);
            __syncthreads();
            first = sm.item;
        } else {
            if (lane == 0) first = atomicAdd(work, tile);
            first = __shfl_sync(CSS_FULL, first, 0);
        }
        if (first >= nitems) break;
        const int end = min(first + tile, nitems);
        for (int k = first; k < end; ++k) {
            const int item = q.item_list ? q.item_list[k] : k;
            const int jid = q.job_of_item ? q.job_of_item[item] : 0;
            const cssi::GeoJob& J = jobs ? jobs[jid] : job0;
            const int pos = q.src_of_item ? q.src_of_item[item] : item;
            Group<R, PL, TEAM, LK> G{J, g.lay, b, h, e, x, sm, tm, J.order ? J.order[pos] : pos, lane, wid,
                                 TEAM ? (int)threadIdx.x : lane, TEAM ? (int)blockDim.x : 32, __double2float_ru(J.rc), {}};
            if constexpr (LK) G.lk.p = reinterpret_cast<Link*>(x + g.lay.s_bytes);
            if constexpr (!TEAM) { G.wid = 0; }
            G.run(item, q.defer_list, q.defer_count, status, counters);
            G.bar();
        }
    }
}

}  // namespace

namespace cssi {

namespace {

// byte offsets of one group's working memory for the given capacities (s_cap 0: no spill area)
template <class R>
WaveLay lay_out(int ring_log, int s_cap, int vh_log, int th_log, bool shared, bool team) {
    WaveLay y{};
    y.r_mask = (1 << ring_log) - 1;
    y.s_cap = s_cap;
    y.vh_log = vh_log;
    y.th_log = th_log;
    const int RG = 1 << ring_log, VH = 1 << vh_log, TH = 1 << th_log, ix = shared ? 2 : 4;
    y.v_most = VH - VH / 8;
    y.t_most = TH - TH / 8;
    y.i_cap = VH * 5 / 16;
    y.lg_cap = team ? 2 * TH : 0;
    int o = 0;
    auto take = [&](int n, int size) {
        const int p = o;
        o = (o + n * size + 15) & ~15;
        return p;
    };
    auto record = [&](int* to, int n) {
        for (int k = 0; k < 5; ++k) to[k] = take(n, 16);
        to[5] = take(n, 2 * ix);
    };
    record(y.r, RG);
    y.h_bytes = o;
    o = 0;
    y.vkey = take(VH, 4); y.vdist = take(VH, 8); y.vinfo = take(VH, ix);
    // 3 TH ints, used once the source is done: in the place of the vertex keys where they fit
    y.tlist = 3 * TH <= VH ? y.vkey : take(3 * TH, 4);
    y.itan = take(y.i_cap, 2 * sizeof(R)); y.iback = take(y.i_cap, 4); y.ihc = take(y.i_cap, 4);
    y.emit = take(2 * y.i_cap, ix);
    y.tkey = take(TH, 4); y.tdist = take(TH, 8); y.tvert = take(sizeof(R) == 4 ? TH : 0, 8);
    const int recs = team ? y.lg_cap : (sizeof(R) == 4 ? 2 * TH : TH);
    y.ttan = take(recs, 2 * sizeof(R));
    y.ldist = take(y.lg_cap, 8); y.lslot = take(y.lg_cap, 4);
    y.t_bytes = o;
    o = 0;
    record(y.s, s_cap);
    y.s_bytes = o;
    o = 0;
    record(y.e, EV);
    y.e_task = take(64, 1);
    y.e_bytes = o;
    return y;
}

int log2_up(int x) {
    int l = 5;
    while ((1 << l) < x) ++l;
    return l;
}

template <class R, int PL, bool TEAM, bool LK>
int blocks_of(int warps, size_t dyn) {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, k_waves<R, PL, TEAM, LK>) != cudaSuccess) { cudaGetLastError(); return 0; }
    const int room = optin - (int)fa.sharedSizeBytes;
    if (dyn > (size_t)room) return 0;
    if (cudaFuncSetAttribute(k_waves<R, PL, TEAM, LK>, cudaFuncAttributeMaxDynamicSharedMemorySize, room) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_waves<R, PL, TEAM, LK>, 32 * warps, dyn) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb;
}

size_t dyn_bytes(const WaveLay& y, int warps, bool shared, bool team) {
    return (size_t)(team ? 1 : warps) * (y.h_bytes + (shared ? y.t_bytes : 0)) + (size_t)warps * y.e_bytes;
}

}  // namespace

// Capacities of one source's working memory.  The ring holds 64 waiting windows in shared memory
// (a team's 128 a warp, 64 in the FP32 form beside tables in shared memory), the rest of half the
// windows waits in a spill area in global memory.
// Tables in shared memory: 256 vertices (a team's 1024) and 64 targets (256) times the scale; in
// global memory they follow the table capacity (0: the windows).  A team's tables and ring are
// halved until the shape fits an SM.
// 64 slots: a small patch has 60-100 windows waiting (CPU counts: 71 icosphere, 101 noisy sphere at
// most), a wave takes 32 and makes as many; 14 KB a warp in all then leave room for 16 warps.
// FP32 teams of 8 with 64 slots a warp go two to an SM (200 sources with 400 faces each on a smooth sphere
// 0.130 ms, 0.226 with 128 slots; 300 with 1000 0.322, 0.466; 100 with 1000 0.261, 0.234).
WaveLay wave_layout(int precision, int win_cap, int tab_cap, int shared_scale, int warps, int team) {
    const bool f32 = precision == CSS_FP32;
    const int tab = tab_cap > 0 ? tab_cap : win_cap;
    int wait = win_cap / 2;
    if (!shared_scale) wait = std::min(wait, std::max(32, tab / 4));
    int rl = std::min(log2_up(wait), team ? log2_up((f32 && shared_scale ? 64 : 128) * warps) : 6);
    int vl = shared_scale ? log2_up((team ? 1024 : 256) * shared_scale) : log2_up(std::max(64, tab / 2));
    int tl = shared_scale ? log2_up((team ? 256 : 64) * shared_scale) : log2_up(std::max(64, tab / 4));
    WaveLay y;
    for (;;) {
        const int spill = wait > (1 << rl) ? 1 << log2_up(wait) : 0;
        y = f32 ? lay_out<float>(rl, spill, vl, tl, shared_scale != 0, team != 0)
                : lay_out<double>(rl, spill, vl, tl, shared_scale != 0, team != 0);
        if (dyn_bytes(y, warps, shared_scale != 0, team != 0) <= WAVE_SHARED_MAX || !team) break;
        if (shared_scale && vl > log2_up(256 * shared_scale)) { --vl; --tl; }
        else if (rl > 6) --rl;
        else break;
    }
    y.max_waves = 4096 + 8 * win_cap;
    return y;
}

WaveLay wave_layout_of(int precision, int spill_log, int vh_log, int th_log) {
    WaveLay y = precision == CSS_FP32 ? lay_out<float>(6, 1 << spill_log, vh_log, th_log, false, false)
                                      : lay_out<double>(6, 1 << spill_log, vh_log, th_log, false, false);
    y.max_waves = 4096 + (64 << spill_log);
    return y;
}

size_t waves_global_bytes(const WaveLay& y, int shared) { return (size_t)y.s_bytes + (shared ? 0 : y.t_bytes); }

int waves_blocks_per_sm(int precision, const WaveLay& y, int warps, int shared, int team) {
    if (warps < 1 || warps > MAXW) return 0;
    const size_t dyn = dyn_bytes(y, warps, shared != 0, team != 0);
#define CSS_PICK(F)                                                                                        \
    (precision == CSS_FP32 ? (shared ? (team ? F<float, 1, true, false>(warps, dyn) : F<float, 1, false, false>(warps, dyn))     \
                                     : (team ? F<float, 0, true, false>(warps, dyn) : F<float, 0, false, false>(warps, dyn)))    \
                           : (shared ? (team ? F<double, 1, true, false>(warps, dyn) : F<double, 1, false, false>(warps, dyn))   \
                                     : (team ? F<double, 0, true, false>(warps, dyn) : F<double, 0, false, false>(warps, dyn))))
    return CSS_PICK(blocks_of);
#undef CSS_PICK
}

cudaError_t launch_waves(const GeoJob& job0, const GeoJob* djobs, const GeoQueue& q, int precision, const WaveWs& g,
                         int warps, int nctas, int* work_counter, int* status, unsigned long long* counters,
                         cudaStream_t st) {
    const size_t dyn = dyn_bytes(g.lay, warps, g.shared != 0, g.team != 0);
#define CSS_LAUNCH(RT, P, T) \
    k_waves<RT, P, T, false><<<nctas, 32 * warps, dyn, st>>>(job0, djobs, q, g, work_counter, status, counters)
    if (precision == CSS_FP32) {
        if (g.shared) { if (g.team) CSS_LAUNCH(float, 1, true); else CSS_LAUNCH(float, 1, false); }
        else { if (g.team) CSS_LAUNCH(float, 0, true); else CSS_LAUNCH(float, 0, false); }
    } else {
        if (g.shared) { if (g.team) CSS_LAUNCH(double, 1, true); else CSS_LAUNCH(double, 1, false); }
        else { if (g.team) CSS_LAUNCH(double, 0, true); else CSS_LAUNCH(double, 0, false); }
    }
#undef CSS_LAUNCH
    return cudaGetLastError();
}

size_t waves_link_bytes(const WaveLay& y) { return sizeof(Link) * (((size_t)1 << y.vh_log) + ((size_t)1 << y.th_log)); }

cudaError_t launch_waves_links(const GeoJob& job, const GeoQueue& q, const WaveWs& g, int warps, int nctas,
                               int* work_counter, int* status, unsigned long long* counters, cudaStream_t st) {
    const size_t dyn = dyn_bytes(g.lay, warps, g.shared != 0, false);
    if ((g.shared ? blocks_of<double, 1, false, true>(warps, dyn) : blocks_of<double, 0, false, true>(warps, dyn)) < 1)
        return cudaErrorInvalidConfiguration;
    if (g.shared) k_waves<double, 1, false, true><<<nctas, 32 * warps, dyn, st>>>(job, nullptr, q, g, work_counter, status, counters);
    else k_waves<double, 0, false, true><<<nctas, 32 * warps, dyn, st>>>(job, nullptr, q, g, work_counter, status, counters);
    return cudaGetLastError();
}

}  // namespace cssi
