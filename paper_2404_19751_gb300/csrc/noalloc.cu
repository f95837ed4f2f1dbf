// noalloc.cu -- allocation-free force evaluation.
//
// Some callers cannot call cudaMalloc at the point where they need forces: code running
// inside a host callback or a framework that forbids device allocation on its hot path,
// or an embedding that must not change the device memory footprint after start-up. For
// them css_compute_forces_noalloc runs the same neighbour/force kernel as
// css_compute_forces, but all of its scratch (the per-warp tables, the face buckets and the launch
// counters) lives in the one file-scope device array below, of a fixed size that every GPU
// loading this library holds until the process exits.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <string>

#include "css_internal.h"

namespace {

constexpr size_t NA_WS_BYTES = 48ull << 20;        // working memory in global memory
constexpr int64_t NA_MAX_FACES = 1 << 20;
constexpr int64_t NA_MAX_PARTICLES = 1 << 18;
constexpr int NA_WARPS_PER_CTA = 4;
constexpr size_t NA_OFF_FCNT = NA_WS_BYTES;
constexpr size_t NA_OFF_FSTART = NA_OFF_FCNT + (NA_MAX_FACES + 1) * 4;
constexpr size_t NA_OFF_FITEMS = NA_OFF_FSTART + (NA_MAX_FACES + 1) * 4;
constexpr size_t NA_OFF_SCAN = NA_OFF_FITEMS + NA_MAX_PARTICLES * 4;
constexpr size_t NA_SCAN_INTS = (NA_MAX_FACES + 1) / 2048 + 2;
constexpr size_t NA_OFF_PCNT = NA_OFF_SCAN + NA_SCAN_INTS * 4;
constexpr size_t NA_OFF_DEFER = NA_OFF_PCNT + NA_MAX_PARTICLES * 4;   // two lists of sources left to a later pass
constexpr size_t NA_OFF_SCAL = (NA_OFF_DEFER + 2 * NA_MAX_PARTICLES * 4 + 255) & ~(size_t)255;  // work, status
constexpr size_t NA_OFF_COUNT = NA_OFF_SCAL + 256;                                              // 8 counters
constexpr size_t NA_BYTES = NA_OFF_COUNT + 8 * 8;   // 62.9 MB in all

static __device__ __align__(256) unsigned char g_noalloc_scratch[NA_BYTES];

struct NaDevice {
    char* base = nullptr;   // device address of g_noalloc_scratch on this device
    int bps[2] = {0, 0};    // resident CTAs per SM of the shared-memory pass, by precision
    bool zeroed = false;    // the face counts start from zero (every call leaves them so)
};
NaDevice g_na[64];

// The caller's particle arrays are checked on the device before any kernel indexes with
// them: a face index outside [0, nf), or a barycentric triple that is not finite, has an
// entry below -1e-12 or does not sum to 1 within 1e-9 (the rule css_particles_set applies
// on the host), sets ST_BAD_INPUT and nothing else runs.
__global__ void k_na_validate(int32_t n, int32_t nf, const int32_t* face, const double* bary, int* status) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int32_t f = face[i];
    const double a = bary[3 * (size_t)i], b = bary[3 * (size_t)i + 1], c = bary[3 * (size_t)i + 2];
    const bool ok = f >= 0 && f < nf && isfinite(a) && isfinite(b) && isfinite(c) && a >= -1e-12 && b >= -1e-12 &&
                    c >= -1e-12 && fabs(a + b + c - 1.0) <= 1e-9;
    if (!ok) atomicOr(status, css::ST_BAD_INPUT);
}

// the current device for the lifetime of the guard, then the caller's again
struct DeviceGuard {
    int prev = -1;
    cudaError_t set(int dev) {
        cudaError_t e = cudaGetDevice(&prev);
        if (e != cudaSuccess) { prev = -1; return e; }
        if (prev == dev) { prev = -1; return cudaSuccess; }
        e = cudaSetDevice(dev);
        if (e != cudaSuccess) prev = -1;
        return e;
    }
    ~DeviceGuard() { if (prev >= 0) cudaSetDevice(prev); }
};

// status bits of the kernel -> C ABI code and message
int na_status_error(css_ctx* c, int status) {
    if (status & css::ST_BAD_INPUT) {
        c->err = "compute_forces_noalloc: a face index is out of range or a barycentric triple is not finite, "
                 "non-negative and summing to 1";
        return CSS_ERR_INVALID_ARG;
    }
    if (status & (css::ST_WIN_OVERFLOW | css::ST_HASH_OVERFLOW)) {
        c->err = "compute_forces_noalloc: a source needs more than the fixed workspace; use css_compute_forces";
        return CSS_ERR_QUEUE_OVERFLOW;
    }
    if (status & (css::ST_ITER_LIMIT | css::ST_WALK_LIMIT)) {
        c->err = "compute_forces_noalloc: a device loop reached its iteration cap";
        return CSS_ERR_ITER_LIMIT;
    }
    c->err = "compute_forces_noalloc: device status " + std::to_string(status);
    return CSS_ERR_CUDA;
}

}  // namespace

int css_compute_forces_noalloc(const css_mesh* mesh, int64_t n, const int32_t* face, const double* bary,
                               const css_potential* pot, double r_c, int precision, double* forces,
                               double* e_pot, void* stream) {
    if (!mesh || !face || !bary || !pot || !forces || n < 1 || !(r_c > 0.0) ||
        (precision != CSS_FP64 && precision != CSS_FP32) || pot->kind < 0 || pot->kind > 2)
        return CSS_ERR_INVALID_ARG;
    css_ctx* c = mesh->ctx;
    if (n > NA_MAX_PARTICLES || mesh->nf > NA_MAX_FACES) {
        c->err = "compute_forces_noalloc: at most " + std::to_string(NA_MAX_PARTICLES) + " particles and " +
                 std::to_string(NA_MAX_FACES) + " faces fit its fixed scratch";
        return CSS_ERR_CAPACITY;
    }
    // everything runs on the device of the mesh's context, whatever device is current
    const int dev = c->device;
    if (dev < 0 || dev >= 64) return CSS_ERR_INVALID_ARG;
    DeviceGuard guard;
    cudaError_t e = guard.set(dev);
    if (e != cudaSuccess) { c->err = std::string("compute_forces_noalloc: ") + cudaGetErrorString(e); return CSS_ERR_CUDA; }
    cudaStream_t st = (cudaStream_t)stream;
    if (st) {   // a stream of another device would put these launches beside the wrong memory
        int sdev = -1;
        e = cudaStreamGetDevice(st, &sdev);
        if (e != cudaSuccess) { cudaGetLastError(); c->err = "compute_forces_noalloc: stream not usable"; return CSS_ERR_INVALID_ARG; }
        if (sdev != dev) {
            c->err = "compute_forces_noalloc: the stream belongs to device " + std::to_string(sdev) +
                     ", the mesh to device " + std::to_string(dev);
            return CSS_ERR_INVALID_ARG;
        }
    }
    NaDevice& D = g_na[dev];
    if (!D.base) {   // first call on this device: host code needs the array's device address
        e = cudaGetSymbolAddress((void**)&D.base, g_noalloc_scratch);
        if (e != cudaSuccess) { D.base = nullptr; c->err = std::string("noalloc set-up: ") + cudaGetErrorString(e); return CSS_ERR_CUDA; }
    }
    int32_t* fcnt = (int32_t*)(D.base + NA_OFF_FCNT);
    int32_t* fstart = (int32_t*)(D.base + NA_OFF_FSTART);
    int32_t* fitems = (int32_t*)(D.base + NA_OFF_FITEMS);
    int32_t* scan = (int32_t*)(D.base + NA_OFF_SCAN);
    int32_t* pcnt = (int32_t*)(D.base + NA_OFF_PCNT);
    int* scal = (int*)(D.base + NA_OFF_SCAL);
    unsigned long long* cnt = (unsigned long long*)(D.base + NA_OFF_COUNT);
    // work already queued on the context's stream (an update or a step writing the arrays
    // read here) comes first; the event was made with the context, so nothing is allocated
    e = cudaEventRecord(c->ev_order, c->stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(st, c->ev_order, 0);
    if (e == cudaSuccess && !D.zeroed) {
        e = cudaMemsetAsync(fcnt, 0, (NA_MAX_FACES + 1) * 4, st);
        if (e == cudaSuccess) D.zeroed = true;
    }
    if (e == cudaSuccess) e = cudaMemsetAsync(scal, 0, 256 + 8 * 8, st);
    int status = 0;
    // the inputs are checked before any kernel indexes with them
    if (e == cudaSuccess) {
        k_na_validate<<<(unsigned)((n + 255) / 256), 256, 0, st>>>((int32_t)n, (int32_t)mesh->nf, face, bary, scal + 1);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&status, scal + 1, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) { c->err = std::string("compute_forces_noalloc: ") + cudaGetErrorString(e); return CSS_ERR_CUDA; }
    if (status) return na_status_error(c, status);
    if (e_pot) e = cudaMemsetAsync(e_pot, 0, sizeof(double), st);
    if (e == cudaSuccess)
        // the pair-count region doubles as the scatter scratch: the kernel below rewrites it
        e = cssi::launch_bucket((int32_t)n, (int32_t)mesh->nf, face, mesh->frank, fcnt, fstart, fitems, pcnt, scan, nullptr, nullptr,
                                st);
    cssi::GeoJob j{};
    j.m = mesh->view();
    j.n = (int32_t)n;
    j.face = face;
    j.bary = bary;
    j.fstart = fstart;
    j.order = fitems;
    j.fitems = fitems;
    j.rc = mesh->in_units(r_c);
    j.pcnt = pcnt;
    j.want_forces = 1;
    j.pot = *pot;
    j.force = forces;
    j.epot = e_pot;
    // three passes, each over the sources the one before could not hold: shared-memory tables; the
    // scratch array in slices for up to 1792 vertices and 896 targets; the same array in fewer
    // slices that hold every particle as a target.  What overflows the last one is reported.
    int32_t* defer = (int32_t*)(D.base + NA_OFF_DEFER);
    for (int pass = 0; pass < 3 && e == cudaSuccess; ++pass) {
        cssi::WaveWs g{};
        g.shared = pass == 0;
        g.base = D.base;
        int tl = 10;
        while (pass == 2 && (7ll << tl) / 8 < n + 1) ++tl;
        g.lay = pass == 0 ? cssi::wave_layout(precision, 256, 0, 1, NA_WARPS_PER_CTA, 0)
                          : cssi::wave_layout_of(precision, pass == 1 ? 10 : 12, pass == 1 ? 11 : 14, tl);
        g.stride = cssi::waves_global_bytes(g.lay, g.shared);
        int warps = NA_WARPS_PER_CTA, ctas = 0;
        if (pass) {
            const int slices = (int)std::min<size_t>(1024, NA_WS_BYTES / g.stride);
            warps = std::min(warps, slices);
            ctas = slices / warps;
        } else {
            int& bps = D.bps[precision];
            if (!bps) bps = cssi::waves_blocks_per_sm(precision, g.lay, warps, 1, 0);
            if (bps < 1) e = cudaErrorInvalidConfiguration;
            ctas = (int)std::min<size_t>((size_t)c->sm_count * bps, NA_WS_BYTES / (g.stride * warps));
        }
        const cssi::GeoQueue q{nullptr, nullptr, (int32_t)n,
                               pass ? defer + (pass - 1) * NA_MAX_PARTICLES : nullptr, pass ? scal + 1 + 2 * pass : nullptr,
                               pass < 2 ? defer + pass * NA_MAX_PARTICLES : nullptr, pass < 2 ? scal + 3 + 2 * pass : nullptr, 1};
        if (e == cudaSuccess)
            e = cssi::launch_waves(j, nullptr, q, precision, g, warps, ctas, pass ? scal + 2 * pass : scal, scal + 1, cnt, st);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&status, scal + 1, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) { c->err = std::string("compute_forces_noalloc: ") + cudaGetErrorString(e); return CSS_ERR_CUDA; }
    if (status) return na_status_error(c, status);
    return CSS_OK;
}
