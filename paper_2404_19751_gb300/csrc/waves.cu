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
// against each window that enters it; the tests are queued and evaluated 32 at a time.
//
// A window's cone is two directions in the frame of its pseudo-source, where they stay what
// they are through every unfolding (the direction to the vertex that bounds the cone), so no
// error builds up and no ray has to be cut with an edge in FP64: the interval on the edge is
// FP32 and rounded outward.  The pseudo-source's image s is FP64 in both forms; the FP32 form
// keeps rotations and directions in FP32.  Lengths of results are FP64 in both forms.
//
// Measured against windows kept in per-edge lists and trimmed against one another (the same
// evaluations, default launch shapes): 65536 particles on a noisy level-8 sphere 110.7 -> 21.7 ms
// (FP64) and 73.1 -> 18.5 ms (FP32), 8192 on a 256 x 256 height field 127 -> 13.9 ms, every pair of
// 64 on a flat plane 30 -> 2.9 ms.  The windows unfolded per source are the same within 10 %
// (482 against 440, 3991 against 3950, 5135 against 5151); a window costs a fifth: no list walk,
// no FP64 split, no local-memory frames.
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

constexpr int MAXW = 8;          // warps per CTA
constexpr int EV = 32;           // queued target tests per warp
constexpr int NONE = -1;
constexpr int FIRST = 1 << 30;   // ring entry: starts at a vertex of the face behind its edge
constexpr int FROM_VERTEX = 1 << 29;   // test: straight from a vertex of the target's face

// relative tolerance of a point on the rim of a cone
template <class R>
struct Rim;
template <>
struct Rim<double> {
    static constexpr double t = 1e-12;
};
template <>
struct Rim<float> {
    static constexpr float t = 2e-6f;
};
// relative excess up to which a window's path is taken over a path from a vertex of the target's face
template <class R>
struct Tie;
template <>
struct Tie<double> {
    static constexpr double t = 1e-13;
};
template <>
struct Tie<float> {
    static constexpr double t = 1e-6;
};

// the counters of one source
struct GroupSm {
    int head, tail;      // first waiting window, end of the ring (both only grow)
    int nem[2], cur;     // vertices waiting to start windows: two lists, the one in use
    unsigned emin;       // a lower bound on their distances (FP32 bits)
    int nv, nt, nlog;    // table entries: vertices, targets, target improvements
    int err;
    int item;
    unsigned nprop;
    float km[MAXW];
    double fx[MAXW], fy[MAXW], en[MAXW];
};

// ------------------------------------------------------------------ working memory
template <class T>
__device__ __forceinline__ T* at(unsigned char* b, int off) { return reinterpret_cast<T*>(b + off); }

__device__ __forceinline__ uint32_t hash_of(int32_t key, int logcap) { return ((uint32_t)key * 2654435761u) >> (32 - logcap); }

__device__ __forceinline__ int tab_find(const int32_t* keys, int logcap, int32_t key) {
    const uint32_t mask = (1u << logcap) - 1u;
    uint32_t s = hash_of(key, logcap);
    for (uint32_t p = 0; p <= mask; ++p) {
        const int32_t c = *(volatile const int32_t*)(keys + s);
        if (c == key) return (int)s;
        if (c == NONE) return NONE;
        s = (s + 1u) & mask;
    }
    return NONE;
}

// slot of the key, claimed if it is new; NONE when the table holds `most` keys already
__device__ __forceinline__ int tab_insert(int32_t* keys, int logcap, int32_t key, int* count, int most, bool& claimed) {
    const uint32_t mask = (1u << logcap) - 1u;
    uint32_t s = hash_of(key, logcap);
    claimed = false;
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

// Where the path through an edge's start vertex (along the edge) stops being the shorter one:
// the window (pseudo-source at (sx, sy) with s2 = |s|^2, sx measured from that vertex) beats it
// for x > x0 only, (x - sx)^2 + sy^2 < (x + a)^2 with a = the vertex's distance minus sigma.
// Rounded so that too little is cut, never too much (eps bounds the rounding of sx); beyond L:
// nothing of the window is left.
__device__ __forceinline__ float cut_at(float sx, float s2, float a, float L, float eps) {
    const float num = s2 - a * a - 2e-6f * (s2 + a * a) - 2.0f * eps * fabsf(sx), den = 2.0f * (a + sx);
    if (!(num > 0.0f)) return 0.0f;
    return den * L > num * 0.999f ? __fdividef(num, den) - 1e-5f * L : 2.0f * L;
}

// Evaluate a warp's queued tests: the target's point in the frame of the entered half-edge, inside
// the cone or not, its length; every improvement of a target's distance is logged with its
// direction at the source (the log is read once the source is done).  Paths that end with a
// straight piece from a vertex of the target's own face are kept apart from those that come
// through a window: a window wins over them unless they are shorter by more than the form's
// precision, so that a direction does not hang on the last bits of two equal lengths.
template <class R>
__device__ __noinline__ void eval_tests(const cssi::GeoJob& J, const WaveLay& Y, unsigned char* b, unsigned char* e,
                                        GroupSm& sm, int nev, int lane) {
    if (lane >= nev) return;
    const DMesh& m = J.m;
    const int he = at<int>(e, Y.e_he)[lane], j = at<int>(e, Y.e_j)[lane];
    int vs = at<int>(e, Y.e_vs)[lane];
    const bool vertex = vs >= 0 && (vs & FROM_VERTEX);
    if (vertex) vs &= ~FROM_VERTEX;
    const double sx = at<double>(e, Y.e_sx)[lane], sy = at<double>(e, Y.e_sy)[lane];
    const R ra = at<R>(e, Y.e_ra)[lane], rb = at<R>(e, Y.e_rb)[lane];
    const R d0x = at<R>(e, Y.e_d0x)[lane], d0y = at<R>(e, Y.e_d0y)[lane];
    const R d1x = at<R>(e, Y.e_d1x)[lane], d1y = at<R>(e, Y.e_d1y)[lane];
    const HeRec& r = m.he[he];
    const int k = he % 3;
    const double* bj = J.bary + 3 * (size_t)j;
    const double bv = bj[k == 2 ? 0 : k + 1], bc = bj[k == 0 ? 2 : k - 1];
    const double gx = bv * r.L + bc * r.cx - sx, gy = bc * r.cy - sy;
    const R fx = (R)gx, fy = (R)gy;
    const R qx = fx * ra + fy * rb, qy = fy * ra - fx * rb;
    const R tol = Rim<R>::t * (R)r.L;
    const bool in = d0x * qy - d0y * qx <= tol * (fabs(d0x) + fabs(d0y)) &&
                    d1x * qy - d1y * qx >= -tol * (fabs(d1x) + fabs(d1y));
    const double n = sqrt(gx * gx + gy * gy), sig = vs < 0 ? 0.0 : at<double>(b, Y.vdist)[vs];
    const double d = sig + n;
    if (!(in && d < J.rc)) return;
    bool claimed;
    const int s = tab_insert(at<int32_t>(b, Y.tkey), Y.th_log, j, &sm.nt, Y.t_most, claimed);
    if (s < 0) {
        atomicOr(&sm.err, css::ST_HASH_OVERFLOW);
        return;
    }
    const unsigned long long bits = (unsigned long long)__double_as_longlong(d);   // lengths start at infinity
    if (atomicMin((unsigned long long*)at<double>(b, vertex ? Y.tvert : Y.tdist) + s, bits) <= bits) return;
    const int l = atomicAdd(&sm.nlog, 1);
    if (l >= Y.lg_cap) {
        atomicOr(&sm.err, css::ST_HASH_OVERFLOW);
        return;
    }
    R tx, ty;
    if (vs < 0) {
        const R inv = n > 0.0 ? (R)1 / (R)n : (R)0;
        tx = qx * inv;
        ty = qy * inv;
    } else {
        tx = at<R>(b, Y.vtan)[2 * vs];
        ty = at<R>(b, Y.vtan)[2 * vs + 1];
    }
    // the length that decides between a window and a vertex: in the FP32 form from FP32
    // coordinates of the target in its face, like every other comparison of that form
    double w = d;
    if constexpr (sizeof(R) == 4) {
        const int f = he / 3;
        const float L01 = m.lay32[3 * f], x2 = m.lay32[3 * f + 1], y2 = m.lay32[3 * f + 2];
        const float px = (float)bj[1] * L01 + (float)bj[2] * x2, py = (float)bj[2] * y2;
        const float ax = k == 0 ? 0.0f : (k == 1 ? L01 : x2), ay = k == 2 ? y2 : 0.0f;
        if (vertex) w = sig + (double)sqrtf((px - ax) * (px - ax) + (py - ay) * (py - ay));
        else {
            const float bx = k == 0 ? L01 : (k == 1 ? x2 : 0.0f), by = k == 1 ? y2 : 0.0f, L = m.he32[he].L;
            const float ex = (bx - ax) / L, ey = (by - ay) / L;
            const float hx = (px - ax) * ex + (py - ay) * ey - (float)sx, hy = ex * (py - ay) - ey * (px - ax) - (float)sy;
            w = (double)((float)sig + sqrtf(hx * hx + hy * hy));
        }
    }
    at<double>(b, Y.ldist)[l] = d;
    at<double>(b, Y.lcmp)[l] = w;
    at<R>(b, Y.ltan)[2 * l] = tx;
    at<R>(b, Y.ltan)[2 * l + 1] = ty;
    at<int>(b, Y.lslot)[l] = vertex ? s | FROM_VERTEX : s;
}

// ------------------------------------------------------------------ one source
template <class R, int PL, bool TEAM>
struct Group {
    const cssi::GeoJob& J;
    const WaveLay& Y;
    unsigned char* b;      // tables and ring
    unsigned char* e;      // this warp's queued tests
    GroupSm& sm;
    int src, lane, wid, tid, T;
    int nev = 0;

    __device__ __forceinline__ void bar() const {
        if constexpr (TEAM) __syncthreads();
        else __syncwarp();
    }
    __device__ __forceinline__ int32_t* vkey() const { return at<int32_t>(b, Y.vkey); }
    __device__ __forceinline__ double* vdist() const { return at<double>(b, Y.vdist); }
    __device__ __forceinline__ R* vtan() const { return at<R>(b, Y.vtan); }
    __device__ __forceinline__ unsigned* vflag() const { return at<unsigned>(b, Y.vflag); }
    __device__ __forceinline__ int32_t* tkey() const { return at<int32_t>(b, Y.tkey); }
    __device__ __forceinline__ double* tdist() const { return at<double>(b, Y.tdist); }
    __device__ __forceinline__ double* tvert() const { return at<double>(b, Y.tvert); }

    __device__ __forceinline__ double dist_of(int32_t v) const {
        const int s = tab_find(vkey(), Y.vh_log, v);
        return s < 0 ? CUDART_INF : *(volatile double*)(vdist() + s);
    }

    __device__ __forceinline__ void eval() {
        __syncwarp();
        if (nev) eval_tests<R>(J, Y, b, e, sm, nev, lane);
        __syncwarp();
        nev = 0;
    }

    // queue the particles of face bucket `key` for the lanes that have one; put(entry) writes
    // the window part of an entry
    template <class Put>
    __device__ __forceinline__ void tests(bool has, int key, Put put) {
        int st = 0, cnt = 0;
        if (has) {
            st = J.fstart[key];
            cnt = J.fstart[key + 1] - st;
        }
        for (int r = 0; __any_sync(CSS_FULL, r < cnt); ++r) {
            int j = src;
            if (r < cnt) j = J.fitems[st + r];
            const unsigned mk = __ballot_sync(CSS_FULL, j != src);
            const int c = __popc(mk);
            if (nev + c > EV) eval();
            if (j != src) {
                const int k = nev + __popc(mk & css::lanemask_lt());
                at<int>(e, Y.e_j)[k] = j;
                put(k);
            }
            nev += c;
        }
    }

    // append windows to the ring (lanes with has); `head` is where the ring's waiting part starts
    struct Win {
        double sx, sy;
        R ra, rb, d0x, d0y, d1x, d1y;
        float b0, b1, key;
        int he, vs;
    };
    __device__ __forceinline__ void push(bool has, const Win& w, int head) {
        const unsigned mk = __ballot_sync(CSS_FULL, has);
        if (!mk) return;
        int base = 0;
        if constexpr (TEAM) {
            if (lane == 0) base = atomicAdd(&sm.tail, __popc(mk));
            base = __shfl_sync(CSS_FULL, base, 0);
        } else {
            base = sm.tail;
            __syncwarp();
            if (lane == 0) sm.tail = base + __popc(mk);
            __syncwarp();
        }
        const int pos = base + __popc(mk & css::lanemask_lt());
        if (has) {
            if (pos - head >= (1 << Y.ring_log)) atomicOr(&sm.err, css::ST_WIN_OVERFLOW);
            else {
                const int s = pos & ((1 << Y.ring_log) - 1);
                at<double>(b, Y.sx)[s] = w.sx;
                at<double>(b, Y.sy)[s] = w.sy;
                at<R>(b, Y.ra)[s] = w.ra;
                at<R>(b, Y.rb)[s] = w.rb;
                at<R>(b, Y.d0x)[s] = w.d0x;
                at<R>(b, Y.d0y)[s] = w.d0y;
                at<R>(b, Y.d1x)[s] = w.d1x;
                at<R>(b, Y.d1y)[s] = w.d1y;
                at<float>(b, Y.b0)[s] = w.b0;
                at<float>(b, Y.b1)[s] = w.b1;
                at<float>(b, Y.key)[s] = w.key;
                at<int>(b, Y.he)[s] = w.he;
                at<int>(b, Y.vs)[s] = w.vs;
            }
        }
    }

    // cut [b0, b1] of an edge of length L by its end vertices' distances du, dv; false if nothing is left
    __device__ __forceinline__ bool cut(float sx, float sy, double sig, double du, double dv, float L, float& b0,
                                        float& b1) const {
        const float sy2 = sy * sy;
        const float tx = L - sx, eps = 2.4e-7f * (fabsf(sx) + L);
        if (du < 1e300) b0 = fmaxf(b0, cut_at(sx, sx * sx + sy2, (float)(du - sig), L, eps));
        if (dv < 1e300) b1 = fminf(b1, L - cut_at(tx, tx * tx + sy2, (float)(dv - sig), L, eps));
        return b1 > b0;
    }
    // a lower bound on the lengths the window carries
    __device__ __forceinline__ float key_of(float sx, float sy, float sig, float b0, float b1) const {
        const float x = fminf(fmaxf(sx, b0), b1) - sx;
        return (sig + sqrtf(x * x + sy * sy)) * (1.0f - 2e-6f) - 2.4e-7f * (fabsf(sx) + b1);
    }

    // a vertex that got a smaller distance: its path's direction at the source and its last leg's
    // direction back; queued for starting windows if it does that and is not queued yet
    __device__ __forceinline__ void improved(int slot, double d, R tx, R ty, float back) {
        vtan()[2 * slot] = tx;
        vtan()[2 * slot + 1] = ty;
        const unsigned f = vflag()[slot];
        vflag()[slot] = (geo::pack_back(back) << 16) | 1u;
        const unsigned dl = __float_as_uint(__double2float_rd(d));
        atomicMin(&sm.emin, dl);
        if (!(f & 1u)) {
            const int p = atomicAdd(&sm.nem[sm.cur], 1);
            if (p < Y.em_cap) at<int>(b, Y.emit)[sm.cur * Y.em_cap + p] = slot;
            else atomicOr(&sm.err, css::ST_HASH_OVERFLOW);
        }
    }

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
    __device__ __forceinline__ void emit(int ne, int head, float kmin);
    __device__ __forceinline__ void wave(int head, int n);
    __device__ __forceinline__ int run(int item, int32_t* defer_list, int* defer_count, int* status,
                                       unsigned long long* counters);
};

// out-of-line entries of the rarely run parts; the group goes by value so that the caller's copy stays
// in registers, its count of queued tests comes back
template <class R, int PL, bool TEAM>
__device__ __noinline__ int call_seed_at_vertex(Group<R, PL, TEAM> g, int hc) {
    g.seed_at_vertex(hc);
    return g.nev;
}
template <class R, int PL, bool TEAM>
__device__ __noinline__ int call_emit(Group<R, PL, TEAM> g, int ne, int head, float kmin) {
    g.emit(ne, head, kmin);
    return g.nev;
}

// Start a source (warp 0): tests for its own face, distances of its corners, one window for
// each edge of its face.
template <class R, int PL, bool TEAM>
__device__ __forceinline__ void Group<R, PL, TEAM>::seed(int f0, double b1, double b2) {
    const DMesh& m = J.m;
    const bool c3 = lane < 3;
    const int h = 3 * f0 + (c3 ? lane : 0);
    const HeRec r = m.he[h];
    // the source from the corner's own weights (no cancellation next to a corner): (hx, hy) in the
    // frame of half-edge h, lx from its end; (ex, ey) the frame's x axis in the face's layout
    const int k0 = h - 3 * f0;
    const double wt[3] = {1.0 - b1 - b2, b1, b2};
    const double wa = k0 == 0 ? wt[0] : (k0 == 1 ? wt[1] : wt[2]), wb = k0 == 0 ? wt[1] : (k0 == 1 ? wt[2] : wt[0]);
    const double wc = k0 == 0 ? wt[2] : (k0 == 1 ? wt[0] : wt[1]);
    const double hx = wb * r.L + wc * r.cx, lx = wa * r.L + wc * (r.L - r.cx), hy = fmax(wc * r.cy, 0.0);
    double ax, ay, bx, by;
    css::face_corner(m, f0, k0, ax, ay);
    css::face_corner(m, f0, k0 + 1, bx, by);
    const double ex = (bx - ax) / r.L, ey = (by - ay) / r.L;
    const double vx = hy * ey - hx * ex, vy = -hy * ex - hx * ey;   // from the source to the corner, in the layout
    tests(lane == 0, m.frank ? m.frank[f0] : f0, [&](int k) {
        at<int>(e, Y.e_he)[k] = h;
        at<int>(e, Y.e_vs)[k] = NONE;
        at<double>(e, Y.e_sx)[k] = hx;
        at<double>(e, Y.e_sy)[k] = hy;
        at<R>(e, Y.e_ra)[k] = (R)1;   // half-edge 0's frame is the layout's
        at<R>(e, Y.e_rb)[k] = (R)0;
        at<R>(e, Y.e_d0x)[k] = at<R>(e, Y.e_d0y)[k] = at<R>(e, Y.e_d1x)[k] = at<R>(e, Y.e_d1y)[k] = (R)0;
    });
    // a source on a corner (to the rounding of its position) has no direction to it: its windows start at the vertex, all around
    const double vd = sqrt(hx * hx + hy * hy);
    const unsigned on = __ballot_sync(CSS_FULL, c3 && vd <= 1e-15 * r.L);
    if (c3 && vd < J.rc && (on == 0 || (on >> lane & 1u))) {
        const int s = vertex(m.fv[h]);
        if (s >= 0) {
            vdist()[s] = vd;
            if (!on && (m.htop[h].x & css::EMITS))
                improved(s, vd, (R)(vx / vd), (R)(vy / vd), geo::back_angle(m, h, ex, ey, -vx, -vy, m.lay[3 * f0]));
        }
    }
    __syncwarp();
    if (on) {
        nev = call_seed_at_vertex<R, PL, TEAM>(*this, 3 * f0 + __ffs(on) - 1);
        return;
    }
    const int tw = m.twin[h];
    Win w;
    w.he = tw;
    w.vs = NONE;
    w.sx = lx;   // the twin runs from the edge's end to its start
    w.sy = -hy;
    w.ra = (R)-ex;
    w.rb = (R)ey;
    w.d0x = (R)(lx * ex + hy * ey);
    w.d0y = (R)(lx * ey - hy * ex);
    w.d1x = (R)vx;
    w.d1y = (R)vy;
    w.b0 = 0.0f;
    w.b1 = (float)r.L;
    w.key = key_of((float)w.sx, (float)w.sy, 0.0f, w.b0, w.b1);
    push(c3 && tw >= 0 && w.key < J.rc, w, 0);
}

// A source on corner hc's vertex: one window opposite each corner of the vertex's ring, tests for
// the ring's faces, and the ring's vertices along its edges.  Directions come from unfolding
// the ring from the source's face, counter-clockwise for the first half and clockwise for the
// rest (at a vertex the direction in the source face's plane depends on that choice).  Serial:
// this is rare.
template <class R, int PL, bool TEAM>
__device__ __forceinline__ void Group<R, PL, TEAM>::seed_at_vertex(int hc) {
    const DMesh& m = J.m;
    const int32_t v = m.fv[hc];
    const int deg = m.ring_start[v + 1] - m.ring_start[v];
    const int f0 = hc / 3;
    double ax, ay, bx, by;
    css::face_corner(m, f0, hc - 3 * f0, ax, ay);
    css::face_corner(m, f0, hc - 3 * f0 + 1, bx, by);
    const double phi0 = atan2(by - ay, bx - ax);
    const int half = m.bnd[v] ? deg : (deg + 1) / 2;
    int left = deg;
#pragma unroll 1
    for (int dir = 0; dir < 2; ++dir) {
        int h = hc;
        double phi = phi0;   // direction of corner h's first edge in the source face's layout
        for (int q = 0; q < (dir == 0 ? half : deg) && left > 0; ++q) {
            if (q > 0 || dir == 1) {
                if (dir == 0) {   // the next corner, across this corner's last edge
                    const int f = h / 3, k = h - 3 * f;
                    const HeRec& a = m.he[h];
                    phi += atan2(a.cy, a.cx);
                    h = m.twin[3 * f + (k == 0 ? 2 : k - 1)];
                    if (h < 0) break;
                } else {          // the corner across this corner's first edge
                    const int o = m.twin[h];
                    if (o < 0) break;
                    const int g = o / 3, kg = o - 3 * g;
                    h = 3 * g + (kg == 2 ? 0 : kg + 1);
                    const HeRec& a = m.he[h];
                    phi -= atan2(a.cy, a.cx);
                }
                if (h == hc) break;
            }
            --left;
            const int fh = h / 3, kh = h - 3 * fh;
            const HeRec r = m.he[h];
            const double co = cos(phi), si = sin(phi);
            tests(lane == 0 && h != hc, m.frank ? m.frank[fh] : fh, [&](int t) {
                at<int>(e, Y.e_he)[t] = h;
                at<int>(e, Y.e_vs)[t] = NONE;
                at<double>(e, Y.e_sx)[t] = at<double>(e, Y.e_sy)[t] = 0.0;
                at<R>(e, Y.e_ra)[t] = (R)co;
                at<R>(e, Y.e_rb)[t] = (R)-si;
                at<R>(e, Y.e_d0x)[t] = at<R>(e, Y.e_d0y)[t] = at<R>(e, Y.e_d1x)[t] = at<R>(e, Y.e_d1y)[t] = (R)0;
            });
            const double ang = atan2(r.cy, r.cx), lc = sqrt(r.cx * r.cx + r.cy * r.cy);
            if (lane < 2) {   // the two other corners of the face, along its edges from the vertex
                const int hn = lane == 0 ? 3 * fh + (kh == 2 ? 0 : kh + 1) : 3 * fh + (kh == 0 ? 2 : kh - 1);
                const double d = lane == 0 ? r.L : lc, a = lane == 0 ? phi : phi + ang;
                if (d < J.rc) {
                    const int s = vertex(m.fv[hn]);
                    if (s >= 0) {
                        const unsigned long long bits = (unsigned long long)__double_as_longlong(d);
                        const unsigned long long old = atomicMin((unsigned long long*)(vdist() + s), bits);
                        if (old > bits && (m.htop[hn].x & css::EMITS))
                            improved(s, d, (R)cos(a), (R)sin(a), __int_as_float(0x7fffffff));
                    }
                }
            }
            __syncwarp();
            const int hop = 3 * fh + (kh == 2 ? 0 : kh + 1);
            Win w;
            w.he = m.twin[hop];
            w.vs = NONE;
            const HeRec o = m.he[hop];
            w.sx = o.L - o.cx;
            w.sy = -o.cy;
            // the twin's x axis runs from the face's far corner c to the first edge's end
            const double tx = (r.L - r.cx) / o.L, ty = -r.cy / o.L;
            w.ra = (R)(tx * co - ty * si);
            w.rb = (R)-(tx * si + ty * co);
            w.d0x = (R)(r.cx * co - r.cy * si);
            w.d0y = (R)(r.cx * si + r.cy * co);
            w.d1x = (R)(r.L * co);
            w.d1y = (R)(r.L * si);
            w.b0 = 0.0f;
            w.b1 = (float)o.L;
            w.key = key_of((float)w.sx, (float)w.sy, 0.0f, w.b0, w.b1);
            push(lane == 0 && w.he >= 0 && w.key < J.rc, w, 0);
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
template <class R, int PL, bool TEAM>
__device__ __forceinline__ void Group<R, PL, TEAM>::emit(int ne, int head, float kmin) {
    const DMesh& m = J.m;
    const int from = sm.cur, to = 1 - from;
    bar();
    if (tid == 0) {
        sm.nem[to] = 0;
        sm.cur = to;
        sm.emin = 0x7f800000u;
    }
    bar();
    for (int base = tid - lane; base < ne; base += T) {
        const int it = base + lane;
        int vs = 0;
        bool go = false;
        double dv = 0.0;
        if (it < ne) {
            vs = at<int>(b, Y.emit)[from * Y.em_cap + it];
            dv = vdist()[vs];
            go = dv <= (double)kmin;
            if (!go) {
                at<int>(b, Y.emit)[to * Y.em_cap + atomicAdd(&sm.nem[to], 1)] = vs;
                atomicMin(&sm.emin, __float_as_uint(__double2float_rd(dv)));
            }
        }
        int rs = 0, len = 0;
        float lo = -INFINITY, hi = INFINITY, th = 0.0f;
        if (go) {
            const unsigned fl = vflag()[vs];
            vflag()[vs] = fl & ~1u;
            const int vid = vkey()[vs];
            rs = m.ring_start[vid];
            len = m.ring_start[vid + 1] - rs;
            if ((fl >> 16) != 0xffffu) {
                th = (float)m.theta[vid];
                const float bk = geo::unpack_back(fl >> 16);
                lo = bk + 3.14159265f - geo::SHADOW_TOL;
                lo -= th * floorf(lo / th);
                hi = lo + (th - 6.28318531f + 2.0f * geo::SHADOW_TOL);
            }
        }
        // one lane per (vertex, corner)
        const int incl = geo::warp_incl_scan(len, lane);
        const int total = __shfl_sync(CSS_FULL, incl, 31);
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
            tests(hit, hit ? m.htop[hc].w : 0, [&](int k) {
                at<int>(e, Y.e_he)[k] = hc;
                at<int>(e, Y.e_vs)[k] = o_vs | FROM_VERTEX;
                at<double>(e, Y.e_sx)[k] = at<double>(e, Y.e_sy)[k] = 0.0;
                at<R>(e, Y.e_ra)[k] = (R)1;
                at<R>(e, Y.e_rb)[k] = (R)0;
                at<R>(e, Y.e_d0x)[k] = at<R>(e, Y.e_d0y)[k] = at<R>(e, Y.e_d1x)[k] = at<R>(e, Y.e_d1y)[k] = (R)0;
            });
            Win w;
            bool ok = false;
            if (hit) {
                const int k = hc - 3 * f, hop = 3 * f + (k == 2 ? 0 : k + 1);
                w.he = m.twin[hop];
                if (w.he >= 0) {
                    const HeRec r = m.he[hop];
                    const float L = (float)r.L;
                    w.vs = o_vs | FIRST;
                    w.sx = r.L - r.cx;
                    w.sy = -r.cy;
                    w.ra = (R)1;
                    w.rb = (R)0;
                    w.b0 = 0.0f;
                    w.b1 = L;
                    if (o_th != 0.0f) {
                        // where the directions c0 and c1 meet the opposite edge, as a part of it
                        const css::HeRec32 q = m.he32[hc];
                        const float ex = q.cx - q.L, ey = q.cy;
                        if (c0 > 1e-5f) {
                            const float s = sinf(c0), c = cosf(c0);
                            const float x = fminf(fmaxf(q.L * s / (ey * c - ex * s), 0.0f), 1.0f);
                            w.b1 = fminf(L, L * (1.0f - x) + 1e-5f * L);
                        }
                        if (c1 < wid_c - 1e-5f) {
                            const float s = sinf(c1), c = cosf(c1);
                            const float x = fminf(fmaxf(q.L * s / (ey * c - ex * s), 0.0f), 1.0f);
                            w.b0 = fmaxf(0.0f, L * (1.0f - x) - 1e-5f * L);
                        }
                    }
                    w.d0x = (R)((double)w.b0 - w.sx);
                    w.d0y = (R)-w.sy;
                    w.d1x = (R)((w.b1 == L ? r.L : (double)w.b1) - w.sx);
                    w.d1y = (R)-w.sy;
                    const int4 tp = m.htop[w.he];
                    ok = cut((float)w.sx, (float)w.sy, o_dv, dist_of(tp.x & css::VMASK), dist_of(tp.y & css::VMASK), L,
                             w.b0, w.b1);
                    w.key = key_of((float)w.sx, (float)w.sy, (float)o_dv, w.b0, w.b1);
                    ok = ok && w.key < J.rc;
                }
            }
            push(ok, w, head);
        }
    }
}

// Unfold the windows head .. head + n of the ring (at most one per thread).
template <class R, int PL, bool TEAM>
__device__ __forceinline__ void Group<R, PL, TEAM>::wave(int head, int n) {
    const DMesh& m = J.m;
    const bool on = tid < n;
    const int s = (head + tid) & ((1 << Y.ring_log) - 1);
    const int he = on ? at<int>(b, Y.he)[s] : 0;
    const int4 tp = m.htop[he];
    tests(on, tp.w, [&](int k) {
        at<int>(e, Y.e_he)[k] = he;
        const int v = at<int>(b, Y.vs)[s];
        at<int>(e, Y.e_vs)[k] = v < 0 ? v : v & ~FIRST;
        at<double>(e, Y.e_sx)[k] = at<double>(b, Y.sx)[s];
        at<double>(e, Y.e_sy)[k] = at<double>(b, Y.sy)[s];
        at<R>(e, Y.e_ra)[k] = at<R>(b, Y.ra)[s];
        at<R>(e, Y.e_rb)[k] = at<R>(b, Y.rb)[s];
        at<R>(e, Y.e_d0x)[k] = at<R>(b, Y.d0x)[s];
        at<R>(e, Y.e_d0y)[k] = at<R>(b, Y.d0y)[s];
        at<R>(e, Y.e_d1x)[k] = at<R>(b, Y.d1x)[s];
        at<R>(e, Y.e_d1y)[k] = at<R>(b, Y.d1y)[s];
    });
    const HeRec r = m.he[he];
    const css::HeRec32 q = m.he32[he];
    const double sx = at<double>(b, Y.sx)[s], sy = at<double>(b, Y.sy)[s];
    const R ra = at<R>(b, Y.ra)[s], rb = at<R>(b, Y.rb)[s];
    const R d0x = at<R>(b, Y.d0x)[s], d0y = at<R>(b, Y.d0y)[s], d1x = at<R>(b, Y.d1x)[s], d1y = at<R>(b, Y.d1y)[s];
    float b0 = at<float>(b, Y.b0)[s], b1 = at<float>(b, Y.b1)[s];
    int vs = at<int>(b, Y.vs)[s];
    const bool first = on && vs >= 0 && (vs & FIRST);
    if (vs >= 0) vs &= ~FIRST;
    if (!on) vs = NONE;
    bar();   // the ring's slots up to head + n are free from here on
    const int head2 = head + n;
    const double sig = vs < 0 ? 0.0 : vdist()[vs];
    const float fsx = (float)sx, fsy = (float)sy, fsig = (float)sig;
    const int32_t vu = tp.x & css::VMASK, vv = tp.y & css::VMASK, vc = tp.z & css::VMASK;
    const bool act = on && cut(fsx, fsy, sig, dist_of(vu), dist_of(vv), q.L, b0, b1) &&
                     key_of(fsx, fsy, fsig, b0, b1) < J.rc;
    // the far corner seen from s: gx, gy in this frame, px, py in the pseudo-source's
    const double gx = r.cx - sx, gy = r.cy - sy;
    const R fgx = (R)gx, fgy = (R)gy;
    const R px = fgx * ra + fgy * rb, py = fgy * ra - fgx * rb;
    const float em = 4e-6f * (fabsf(fsx) + fabsf(fsy) + q.L);   // bounds the rounding of FP32 crossings
    const float xc = fsx - (q.cx - fsx) * __fdividef(fsy, q.cy - fsy);
    const R tolg = Rim<R>::t * (R)(fabsf((float)fgx) + fabsf((float)fgy));
    const R t0 = tolg * (fabs(d0x) + fabs(d0y)), t1 = tolg * (fabs(d1x) + fabs(d1y));
    const R cr0 = d0x * py - d0y * px, cr1 = d1x * py - d1y * px;   // < 0: c lies right of the direction
    const bool left = act && cr0 < -t0 && xc > b0 - em, right = act && cr1 > t1 && xc < b1 + em;
    const bool cin = act && cr0 <= t0 && cr1 >= -t1 && xc >= b0 - em && xc <= b1 + em;
    // distance candidates: the far corner, and the two ends of a window that just started
    const int nq = (TEAM ? __syncthreads_or(first) : __any_sync(CSS_FULL, first)) ? 3 : 1;
#pragma unroll 1
    for (int a = 0; a < nq; ++a) {
        bool has = a == 0 ? cin : (first && act && (a == 1 ? b0 <= 0.0f : b1 >= q.L));
        const double vx = a == 0 ? gx : (a == 1 ? -sx : r.L - sx), vy = a == 0 ? gy : -sy;
        const int vtop = a == 0 ? tp.z : (a == 1 ? tp.x : tp.y);
        const float fd = fsig + sqrtf((float)vx * (float)vx + (float)vy * (float)vy);
        int slot = NONE;
        unsigned long long bits = 0, old = 0;
        double d = 0.0;
        if (has && (double)fd * (1.0 - 1e-6) < J.rc) {
            slot = vertex(vtop & css::VMASK);
            if (slot >= 0 && (double)fd * (1.0 - 1e-6) < *(volatile double*)(vdist() + slot)) {
                // the other vertices' distances only cut windows: an FP32 upper bound will do
                d = (vtop & css::EMITS) ? sig + sqrt(vx * vx + vy * vy) : (double)(fd * (1.0f + 1e-6f));
                bits = (unsigned long long)__double_as_longlong(d);
                if (d < J.rc) old = atomicMin((unsigned long long*)(vdist() + slot), bits);
            }
        }
        bar();
        if (old > bits && (vtop & css::EMITS) &&
            *(volatile unsigned long long*)(vdist() + slot) == bits) {
            R tx, ty;
            if (vs < 0) {
                const R inv = (R)1 / (R)d;   // sigma is 0
                tx = px * inv;
                ty = py * inv;
            } else {
                tx = vtan()[2 * vs];
                ty = vtan()[2 * vs + 1];
            }
            const int f = he / 3, k = he - 3 * f;
            const int hc = a == 0 ? 3 * f + (k == 0 ? 2 : k - 1) : (a == 1 ? he : m.twin[he]);
            improved(slot, d, tx, ty,
                     geo::back_angle(m, hc, a == 0 ? -r.cx : (a == 1 ? 1.0 : -1.0), a == 0 ? -r.cy : 0.0, -vx, -vy, r.L));
        }
        bar();
    }
    // the children: side 0 the edge u -> c, side 1 the edge c -> v
    const double du = dist_of(vu), dc = dist_of(vc), dv = dist_of(vv);
#pragma unroll 1
    for (int a = 0; a < 2; ++a) {
        Win w;
        w.he = a == 0 ? r.tl : r.tr;
        bool has = (a == 0 ? left : right) && w.he >= 0;
        if (has) {
            const double co = a == 0 ? r.cl : r.cr, si = a == 0 ? r.sl : r.sr;
            const R fco = sizeof(R) == 4 ? (R)(a == 0 ? q.cl : q.cr) : (R)co, fsi = sizeof(R) == 4 ? (R)(a == 0 ? q.sl : q.sr) : (R)si;
            const double ux = a == 0 ? sx : -gx, uy = a == 0 ? sy : -gy;   // s from the child edge's start
            w.sx = ux * co + uy * si;
            w.sy = uy * co - ux * si;
            if (w.sy > 0.0) w.sy = 0.0;
            w.ra = ra * fco + rb * fsi;
            w.rb = rb * fco - ra * fsi;
            // the corner bounds the child's cone unless it lies beyond the rim on that side
            const bool n0 = a == 1 && cr0 <= t0, n1 = a == 0 && cr1 >= -t1;
            w.d0x = n0 ? px : d0x;
            w.d0y = n0 ? py : d0y;
            w.d1x = n1 ? px : d1x;
            w.d1y = n1 ? py : d1y;
            // the interval: where the rays through b0 and b1 meet the child's edge, rounded outward
            const float ax = a == 0 ? 0.0f : q.cx, ay = a == 0 ? 0.0f : q.cy;
            const float ex = a == 0 ? q.cx : q.L - q.cx, ey = a == 0 ? q.cy : -q.cy;
            const float Lc = sqrtf(ex * ex + ey * ey);
            const float vx = fsx - ax, vy = fsy - ay;
            const float x0 = b0 - fsx, x1 = b1 - fsx;   // ray directions (x, -sy)
            const float m0 = -vx * fsy - vy * x0, e0 = -ex * fsy - ey * x0;
            const float m1 = -vx * fsy - vy * x1, e1 = -ex * fsy - ey * x1;
            // rounding of a crossing: that of the coordinates (em), and that of the ray's direction, which
            // grows as s nears the point the ray goes through
            const float emc = em + 4e-6f * Lc, emd = em * (Lc + q.L);
            const float p0 = emc + __fdividef(emd, fmaxf(fabsf(x0), -fsy)), p1 = emc + __fdividef(emd, fmaxf(fabsf(x1), -fsy));
            w.b0 = a == 1 && xc >= b0 ? 0.0f : fmaxf(0.0f, fminf(e0 != 0.0f ? __fdividef(m0, e0) : 0.0f, 1.0f) * Lc - p0);
            w.b1 = a == 0 && xc <= b1 ? Lc : fminf(Lc, fmaxf(e1 != 0.0f ? __fdividef(m1, e1) : 0.0f, 0.0f) * Lc + p1);
            const float cx = (float)w.sx, cy = (float)w.sy;
            has = cut(cx, cy, sig, a == 0 ? du : dc, a == 0 ? dc : dv, Lc, w.b0, w.b1);
            w.key = key_of(cx, cy, fsig, w.b0, w.b1);
            has = has && w.key < J.rc;
            w.vs = vs;
        }
        push(has, w, head2);
    }
}

template <class R, int PL, bool TEAM>
__device__ __forceinline__ int Group<R, PL, TEAM>::run(int item, int32_t* defer_list, int* defer_count, int* status,
                                                       unsigned long long* counters) {
    const DMesh& m = J.m;
    const int f0 = J.face[src];
    const double* bs = J.bary + 3 * (size_t)src;
    // empty tables; distances start at infinity
    for (int k = tid; k < (1 << Y.vh_log); k += T) {
        vkey()[k] = NONE;
        vdist()[k] = CUDART_INF;
        vflag()[k] = 0;
    }
    for (int k = tid; k < (1 << Y.th_log); k += T) {
        tkey()[k] = NONE;
        tdist()[k] = tvert()[k] = CUDART_INF;
    }
    if (tid == 0) {
        sm.head = sm.tail = sm.nem[0] = sm.nem[1] = sm.cur = sm.nv = sm.nt = sm.nlog = sm.err = 0;
        sm.emin = 0x7f800000u;
    }
    bar();
    if (wid == 0) seed(f0, bs[1], bs[2]);
    unsigned nprop = 0;
    int waves = 0;
    for (;;) {
        bar();
        const int head = sm.head;
        int tail = sm.tail;
        const int ne = sm.nem[sm.cur];
        int err = sm.err;
        if (++waves > Y.max_waves) err |= css::ST_ITER_LIMIT;
        bar();
        if (err || (head == tail && ne == 0)) {
            if (tid == 0) sm.err = err;
            break;
        }
        if (ne > 0) {
            float km = INFINITY;
            tail = min(tail, head + (1 << Y.ring_log));
            for (int k = head + tid; k < tail; k += T) km = fminf(km, at<float>(b, Y.key)[k & ((1 << Y.ring_log) - 1)]);
            km = __uint_as_float(__reduce_min_sync(CSS_FULL, __float_as_uint(km)));
            if constexpr (TEAM) {
                if (lane == 0) sm.km[wid] = km;
                __syncthreads();
                for (int w = 0; w < (T >> 5); ++w) km = fminf(km, sm.km[w]);
            }
            if (head == tail || __uint_as_float(sm.emin) <= km) {
                nev = call_emit<R, PL, TEAM>(*this, ne, head, km);
                bar();
                tail = sm.tail;
            }
        }
        const int n = min(min(tail - head, 1 << Y.ring_log), T);   // a full ring dropped the rest (and reports it)
        wave(head, n);
        nprop += n;
        if (tid == 0) sm.head = head + n;
    }
    eval();
    bar();
    const int err = sm.err;
    if (defer_list && err) {   // a patch too large for this pass: the second pass takes the source
        if (tid == 0) {
            defer_list[atomicAdd(defer_count, 1)] = item;
            atomicAdd(counters + 4, 1ull);
        }
        return 0;
    }
    // the targets in particle order (every sum below runs in that order, so it does not depend on
    // the order of discovery)
    const int nt = sm.nt;
    int* list = at<int>(b, Y.tlist);
    int* ord = list + (1 << Y.th_log);
    if (tid == 0) sm.head = 0;
    bar();
    for (int k = tid; k < (1 << Y.th_log); k += T)
        if (tkey()[k] != NONE) list[atomicAdd(&sm.head, 1)] = k;
    bar();
    if (nt <= 128) {
        for (int k = tid; k < nt; k += T) {
            const int s = list[k], j = tkey()[s];
            int rank = 0;
            for (int q = 0; q < nt; ++q) rank += tkey()[list[q]] < j;
            ord[rank] = s;
        }
    } else {   // bitonic sort
        int n2 = 128;
        while (n2 < nt) n2 <<= 1;
        for (int k = tid; k < n2; k += T) ord[k] = k < nt ? list[k] : NONE;
        bar();
        for (int size = 2; size <= n2; size <<= 1)
            for (int step = size >> 1; step > 0; step >>= 1) {
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
    // the log entries that hold each target's distance through a window and from a vertex
    int* own = list;
    int* ownv = ord + (1 << Y.th_log);
    for (int l = tid; l < min(sm.nlog, Y.lg_cap); l += T) {
        const int s = at<int>(b, Y.lslot)[l] & ~FROM_VERTEX;
        const bool vertex = at<int>(b, Y.lslot)[l] & FROM_VERTEX;
        if (at<double>(b, Y.ldist)[l] == (vertex ? tvert() : tdist())[s]) (vertex ? ownv : own)[s] = l;
    }
    bar();
    double fx = 0.0, fy = 0.0, en = 0.0;
    const double* fr = m.frame + 9 * (size_t)f0;
    for (int k = tid; k < nt; k += T) {
        const int s = ord[k];
        const double dw = tdist()[s], dv = tvert()[s];
        int l = dw < CUDART_INF ? own[s] : ownv[s];
        if (dw < CUDART_INF && dv < dw) {
            const double cw = at<double>(b, Y.lcmp)[l], cv = at<double>(b, Y.lcmp)[ownv[s]];
            if (cv < cw - Tie<R>::t * cv) l = ownv[s];
        }
        const double d = at<double>(b, Y.ldist)[l];
        const double tx = (double)at<R>(b, Y.ltan)[2 * l], ty = (double)at<R>(b, Y.ltan)[2 * l + 1];
        if (J.want_pairs && k < J.pair_cap) {
            const size_t o = (size_t)src * J.pair_cap + k;
            J.pj[o] = tkey()[s];
            J.pd[o] = d;
            J.pt[3 * o] = tx * fr[3] + ty * fr[6];
            J.pt[3 * o + 1] = tx * fr[4] + ty * fr[7];
            J.pt[3 * o + 2] = tx * fr[5] + ty * fr[8];
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
            sm.fx[wid] = fx;
            sm.fy[wid] = fy;
            sm.en[wid] = en;
        }
        __syncthreads();
        if (tid == 0)
            for (int w = 1; w < (T >> 5); ++w) {
                fx += sm.fx[w];
                fy += sm.fy[w];
                en += sm.en[w];
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
        int st = err;
        if (J.want_pairs && nt > J.pair_cap) st |= css::ST_PAIR_OVERFLOW;
        if (st) atomicOr(status, st);
        atomicAdd(counters + 0, 1ull);
        atomicAdd(counters + 1, (unsigned long long)sm.tail);
        atomicAdd(counters + 2, (unsigned long long)nprop);
        atomicAdd(counters + 3, (unsigned long long)nt);
    }
    return 0;
}

// PL 1: tables and ring in shared memory, 0: in the group's slice of global memory.  TEAM: the
// warps of a CTA work on one source, else each warp on its own.  Persistent: groups pull work
// items from a counter.
template <class R, int PL, bool TEAM>
__global__ void __launch_bounds__(256, 2) k_waves(const __grid_constant__ cssi::GeoJob job0, const cssi::GeoJob* jobs,
                                                  const __grid_constant__ cssi::GeoQueue q,
                                                  const __grid_constant__ WaveWs g, int* work, int* status,
                                                  unsigned long long* counters) {
    __shared__ GroupSm sms[TEAM ? 1 : MAXW];
    extern __shared__ __align__(16) unsigned char dsm[];
    const int wpc = blockDim.x >> 5, wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int in_cta = TEAM ? 0 : wid, groups = TEAM ? 1 : wpc;
    GroupSm& sm = sms[in_cta];
    const int gid = blockIdx.x * groups + in_cta;
    unsigned char* b = PL == 1 ? dsm + (size_t)in_cta * g.lay.bytes : (unsigned char*)g.base + (size_t)gid * g.stride;
    unsigned char* e = dsm + (PL == 1 ? (size_t)groups * g.lay.bytes : 0) + (size_t)wid * g.lay.e_bytes;
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
            Group<R, PL, TEAM> G{J, g.lay, b, e, sm, J.order ? J.order[pos] : pos, lane, wid,
                                 TEAM ? (int)threadIdx.x : lane, TEAM ? (int)blockDim.x : 32};
            if constexpr (!TEAM) { G.wid = 0; }
            G.run(item, q.defer_list, q.defer_count, status, counters);
            G.bar();
        }
    }
}

}  // namespace

namespace cssi {

namespace {

// byte offsets of one group's working memory for the given capacities
template <class R>
WaveLay lay_out(int ring_log, int vh_log, int th_log) {
    WaveLay y{};
    y.ring_log = ring_log;
    y.vh_log = vh_log;
    y.th_log = th_log;
    const int RG = 1 << ring_log, VH = 1 << vh_log, TH = 1 << th_log;
    y.v_most = VH - VH / 8;
    y.t_most = TH - TH / 8;
    y.em_cap = VH / 2;
    y.lg_cap = TH + TH / 2;
    int o = 0;
    auto take = [&](int n, int size) {
        const int p = o;
        o = (o + n * size + 15) & ~15;
        return p;
    };
    y.sx = take(RG, 8); y.sy = take(RG, 8);
    y.ra = take(RG, sizeof(R)); y.rb = take(RG, sizeof(R));
    y.d0x = take(RG, sizeof(R)); y.d0y = take(RG, sizeof(R));
    y.d1x = take(RG, sizeof(R)); y.d1y = take(RG, sizeof(R));
    y.b0 = take(RG, 4); y.b1 = take(RG, 4); y.key = take(RG, 4);
    y.he = take(RG, 4); y.vs = take(RG, 4);
    y.vkey = take(VH, 4); y.vdist = take(VH, 8); y.vtan = take(VH, 2 * sizeof(R)); y.vflag = take(VH, 4);
    y.tkey = take(TH, 4); y.tdist = take(TH, 8); y.tvert = take(TH, 8); y.tlist = take(3 * TH, 4);
    y.emit = take(2 * y.em_cap, 4);
    y.ldist = take(y.lg_cap, 8); y.lcmp = take(y.lg_cap, 8); y.ltan = take(y.lg_cap, 2 * sizeof(R)); y.lslot = take(y.lg_cap, 4);
    y.bytes = o;
    o = 0;
    y.e_sx = take(EV, 8); y.e_sy = take(EV, 8);
    y.e_ra = take(EV, sizeof(R)); y.e_rb = take(EV, sizeof(R));
    y.e_d0x = take(EV, sizeof(R)); y.e_d0y = take(EV, sizeof(R));
    y.e_d1x = take(EV, sizeof(R)); y.e_d1y = take(EV, sizeof(R));
    y.e_he = take(EV, 4); y.e_vs = take(EV, 4); y.e_j = take(EV, 4);
    y.e_bytes = o;
    return y;
}

int log2_up(int x) {
    int l = 5;
    while ((1 << l) < x) ++l;
    return l;
}

template <class R, int PL, bool TEAM>
int blocks_of(int warps, size_t dyn) {
    int dev = 0, optin = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    cudaFuncAttributes fa;
    if (cudaFuncGetAttributes(&fa, k_waves<R, PL, TEAM>) != cudaSuccess) { cudaGetLastError(); return 0; }
    const int room = optin - (int)fa.sharedSizeBytes;
    if (dyn > (size_t)room) return 0;
    if (cudaFuncSetAttribute(k_waves<R, PL, TEAM>, cudaFuncAttributeMaxDynamicSharedMemorySize, room) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_waves<R, PL, TEAM>, 32 * warps, dyn) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return nb;
}

size_t dyn_bytes(const WaveLay& y, int warps, bool shared, bool team) {
    return (shared ? (size_t)(team ? 1 : warps) * y.bytes : 0) + (size_t)warps * y.e_bytes;
}

}  // namespace

// Capacities of one source's working memory.  In shared memory: 256 vertices and 64 targets
// times the scale, and a ring of a sixteenth of the windows (a quarter in the team form, whose
// waves are wider), at most 128 times the scale (1024 for a team) and halved until the shape
// fits an SM.  In global memory the tables follow the table capacity (0: the windows).
WaveLay wave_layout(int precision, int win_cap, int tab_cap, int shared_scale, int warps, int team) {
    const int share = team ? win_cap / 4 : win_cap / 16;
    const bool f32 = precision == CSS_FP32;
    auto lay = [&](int r, int v, int t) { return f32 ? lay_out<float>(r, v, t) : lay_out<double>(r, v, t); };
    WaveLay y;
    if (shared_scale) {
        const int most = team ? std::max(1024, 128 * shared_scale) : 128 * shared_scale;
        int rl = log2_up(std::min(share, most));
        const int vl = log2_up(256 * shared_scale), tl = log2_up(64 * shared_scale);
        y = lay(rl, vl, tl);
        while (rl > 5 && dyn_bytes(y, warps, true, team != 0) > WAVE_SHARED_MAX) y = lay(--rl, vl, tl);
    } else {
        const int tab = tab_cap > 0 ? tab_cap : win_cap;
        y = lay(log2_up(std::min(share, std::max(32, tab / 4))), log2_up(std::max(64, tab / 2)), log2_up(std::max(64, tab / 4)));
    }
    y.max_waves = 4096 + 8 * win_cap;
    return y;
}

WaveLay wave_layout_of(int precision, int ring_log, int vh_log, int th_log) {
    WaveLay y = precision == CSS_FP32 ? lay_out<float>(ring_log, vh_log, th_log) : lay_out<double>(ring_log, vh_log, th_log);
    y.max_waves = 4096 + (128 << ring_log);
    return y;
}

int waves_blocks_per_sm(int precision, const WaveLay& y, int warps, int shared, int team) {
    if (warps < 1 || warps > MAXW) return 0;
    const size_t dyn = dyn_bytes(y, warps, shared != 0, team != 0);
#define CSS_PICK(F)                                                                                        \
    (precision == CSS_FP32 ? (shared ? (team ? F<float, 1, true>(warps, dyn) : F<float, 1, false>(warps, dyn))     \
                                     : (team ? F<float, 0, true>(warps, dyn) : F<float, 0, false>(warps, dyn)))    \
                           : (shared ? (team ? F<double, 1, true>(warps, dyn) : F<double, 1, false>(warps, dyn))   \
                                     : (team ? F<double, 0, true>(warps, dyn) : F<double, 0, false>(warps, dyn))))
    return CSS_PICK(blocks_of);
#undef CSS_PICK
}

cudaError_t launch_waves(const GeoJob& job0, const GeoJob* djobs, const GeoQueue& q, int precision, const WaveWs& g,
                         int warps, int nctas, int* work_counter, int* status, unsigned long long* counters,
                         cudaStream_t st) {
    const size_t dyn = dyn_bytes(g.lay, warps, g.shared != 0, g.team != 0);
#define CSS_LAUNCH(RT, P, T) \
    k_waves<RT, P, T><<<nctas, 32 * warps, dyn, st>>>(job0, djobs, q, g, work_counter, status, counters)
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

}  // namespace cssi
