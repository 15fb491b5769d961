// Allocation-free density pass (mdpd_density_noalloc).
//
// Some callers cannot let a library allocate device memory: a plugin inside a
// host application that owns the whole device-memory budget and hands out only
// the input and output buffers, or a caller on a latency-critical path where
// cudaMalloc/cudaFree (which can synchronise the device) are not allowed.  For
// them this file offers one entry point that computes the local densities of a
// set of particles without allocating anything: every temporary buffer of the
// binning and density kernels lives in one file-scope __device__ array of fixed
// size (below), which each GPU that loads the library keeps until the process
// exits.
//
// Host code may not use the array's name as a device address (in host code it
// names a host-side stand-in).  The device address is looked up with
// cudaGetSymbolAddress, with the device current, on every call made outside
// stream capture (so a cudaDeviceReset between calls leaves no stale address);
// a call made while its stream is being captured reuses the address of the
// last uncaptured call on that device, so the first call on a device should
// happen before any stream capture.  All calls share the array and it keeps the previous call's contents,
// so the counters that must start at zero are cleared on every call, and calls
// whose work overlaps on the GPU (on different streams, or from several host
// threads without ordering) race on the array and give wrong results.
//
// A call is short (48,000 particles: 4 MB of traffic, most of it in L2), so it is bound
// by the chain of its launches and by the density kernel.  The binning kernels run next
// to no FP64 (1/64 of the FP32 rate), the tile sums of the scan come from the count, a
// rank per particle takes the place of a sort per cell (one thread sorted a cell while
// the others waited), the density kernel is that of the step (FP16 filter, no lists) and
// writes the caller's order itself, and each kernel's launch overlaps its predecessor's
// end: six device operations instead of nine.  48,000 particles in FP32: 138 -> 80 us.
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>

#include "pair.cuh"

namespace mdpd {

void set_global_error(const std::string& msg);

namespace {

constexpr int64_t NA_MAX_PARTICLES = 65536;
constexpr int64_t NA_MAX_CELLS = 32768;
constexpr size_t NA_ALIGN = 256;

constexpr size_t na_round(size_t b) { return (b + NA_ALIGN - 1) / NA_ALIGN * NA_ALIGN; }

// Byte offsets of the parts of the scratch array.
constexpr size_t OFF_COUNT = 0;
constexpr size_t OFF_SUMS = OFF_COUNT + na_round(NA_MAX_CELLS * 4);      // cleared with the counts
constexpr size_t OFF_START = OFF_SUMS + na_round(64 * 4);
constexpr size_t OFF_CELLOF = OFF_START + na_round((NA_MAX_CELLS + 1) * 4);
constexpr size_t OFF_SLOT = OFF_CELLOF + na_round(NA_MAX_PARTICLES * 4);
constexpr size_t OFF_KEY = OFF_SLOT + na_round(NA_MAX_PARTICLES * 4);
constexpr size_t OFF_SRC = OFF_KEY + na_round(NA_MAX_PARTICLES * 4);
constexpr size_t OFF_CELLS = OFF_SRC + na_round(NA_MAX_PARTICLES * 4);
constexpr size_t OFF_POS4 = OFF_CELLS + na_round(NA_MAX_PARTICLES * 4);
constexpr size_t OFF_FPOS = OFF_POS4 + na_round(NA_MAX_PARTICLES * sizeof(D4));
constexpr size_t OFF_HPOS = OFF_FPOS + na_round(NA_MAX_PARTICLES * sizeof(float4));
constexpr size_t NA_BYTES = OFF_HPOS + na_round(hpos_words(NA_MAX_PARTICLES) * sizeof(uint16_t));

// The scratch memory (about 5.3 MB).
static __device__ __align__(256) unsigned char g_na_scratch[NA_BYTES];

constexpr int NA_MAX_DEVICES = 64;
std::mutex g_na_mutex;
void* g_na_ptr[NA_MAX_DEVICES] = {};

// Device address of the scratch array on the current device.  Outside stream
// capture it is looked up on every call (a lookup allocates nothing), so a
// cudaDeviceReset or a new primary context between calls cannot leave a
// stale address behind; while the stream is being captured the address
// recorded by the last uncaptured call on this device is used, and a call
// that has none is refused.
int scratch_address(cudaStream_t st, void** out, std::string& why)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        why = std::string("cudaGetDevice: ") + cudaGetErrorString(e);
        return MDPD_ERR_CUDA;
    }
    if (dev < 0 || dev >= NA_MAX_DEVICES) {
        why = "device index out of range for the scratch table";
        return MDPD_ERR_INVALID_ARG;
    }
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    e = cudaStreamIsCapturing(st, &cap);
    if (e != cudaSuccess) {
        why = std::string("cudaStreamIsCapturing: ") + cudaGetErrorString(e);
        return MDPD_ERR_CUDA;
    }
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (cap == cudaStreamCaptureStatusNone) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_na_scratch);
        if (e != cudaSuccess || !p) {
            why = std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e);
            return MDPD_ERR_CUDA;
        }
        g_na_ptr[dev] = p;
    } else if (!g_na_ptr[dev]) {
        why = "the first call on a device must come before any stream capture";
        return MDPD_ERR_INVALID_ARG;
    }
    *out = g_na_ptr[dev];
    return MDPD_OK;
}

// Coordinate k of particle i on its way into the lattice: *out is raised if it is not
// finite or, on a non-periodic axis, outside the box (the closed upper face is accepted:
// a particle on it is binned into the last cell, where the search of the neighbouring
// cells stays complete); a periodic one is returned wrapped.  FP64 instructions run
// for the few that need them, under warp-voted branches (see k_load_state).
__device__ __forceinline__ double na_coordinate(const double* __restrict__ pos, int i, int k,
                                                const Geo& geo, bool* out)
{
    double x = pos[3 * (int64_t)i + k];
    const int64_t kx = f64_key(x);
    if (!isfinite(x)) *out = true;
    else if (!geo.periodic[k] && (kx < geo.key_lo[k] || kx > geo.key_hi[k])) *out = true;
    const bool wrap = geo.periodic[k] && isfinite(x) && (kx < geo.key_lo[k] || kx >= geo.key_in[k]);
    if (__any_sync(__activemask(), wrap)) {
        if (wrap) x -= geo.L[k] * floor((x - geo.lo[k]) / geo.L[k]);
    }
    return x;
}

// Cell index along axis k, clamped to the lattice (FP32 away from the cell faces, as in
// k_bin_count).
__device__ __forceinline__ int na_cell(double x, int k, const Geo& geo, const Phys& ph)
{
    const float t = (to_f32(x) - ph.df.lo[k]) * ph.df.inv_h[k];
    const float fl = floorf(t);
    int c = (int)fl;
    const bool exact = ((ph.fast_cell >> k) & 1u) && t - fl > 2e-3f && fl + 1.0f - t > 2e-3f;
    if (__any_sync(__activemask(), !exact)) {
        if (!exact) c = (int)floor_index_f64(x, geo.lo[k], geo.inv_h[k], 0.0, 0);
    }
    return c < 0 ? 0 : (c >= geo.nc[k] ? geo.nc[k] - 1 : c);
}

__global__ void k_na_count(int n, const double* __restrict__ pos, Geo geo, Phys ph,
                           uint32_t* __restrict__ cellof, uint32_t* __restrict__ slot,
                           uint32_t* __restrict__ count, uint32_t* __restrict__ tsum)
{
    pdl_enter();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned act = __ballot_sync(0xffffffffu, i < n);
    if (i >= n) return;
    int q[3];
    bool out = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) q[k] = na_cell(na_coordinate(pos, i, k, geo, &out), k, geo, ph);
    const uint32_t c = (uint32_t)(q[0] + geo.nc[0] * (q[1] + geo.nc[1] * q[2]));
    cellof[i] = c;
    slot[i] = atomicAdd(&count[c], 1u);
    const uint32_t tile = c / (uint32_t)SCAN_TILE;       // the scan's tile sums
    const unsigned peers = __match_any_sync(act, tile);
    if ((threadIdx.x & 31) == (unsigned)(__ffs(peers) - 1))
        atomicAdd(&tsum[tile], (uint32_t)__popc(peers));
}

__global__ void k_na_scatter(int n, const uint32_t* __restrict__ cellof,
                             const uint32_t* __restrict__ slot, const uint32_t* __restrict__ start,
                             uint32_t* __restrict__ key)
{
    pdl_enter();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t d = start[cellof[i]] + slot[i];
    if (d < (uint32_t)n) key[d] = (uint32_t)i;
}

// Order inside each cell by particle index and gather (as k_rank_gather): position as
// offset from the cell centre, the filter's FP16 form, and the particle's index with its
// top bit set if it lies outside the box.
template <typename T>
__global__ void k_na_gather(int n, const double* __restrict__ pos, const uint32_t* __restrict__ key,
                            const uint32_t* __restrict__ cellof, const uint32_t* __restrict__ start,
                            Geo geo, Phys ph, typename Vec4<T>::type* __restrict__ pos4,
                            float4* __restrict__ fpos, uint16_t* __restrict__ hpos,
                            uint32_t* __restrict__ cell_s, uint32_t* __restrict__ src)
{
    pdl_enter();
    const int a = blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= n) return;
    const uint32_t i = key[a];
    if (i >= (uint32_t)n) return;                // (scratch written by an overlapping call)
    const uint32_t c = cellof[i];
    if (c >= (uint32_t)geo.ncell) return;
    const uint32_t b = start[c], e = start[c + 1];
    if (b > e || e > (uint32_t)n) return;
    uint32_t r = 0;
    for (uint32_t q = b; q < e; ++q) r += key[q] < i ? 1u : 0u;
    const uint32_t s = b + r;
    int q[3];
    cell_coords(c, geo, q[0], q[1], q[2]);
    T off[3];
    float fo[3];
    bool out = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double x = na_coordinate(pos, (int)i, k, geo, &out);
        const Derived<float>& f = ph.df;
        float o = 0.0f;
        bool done = sizeof(T) == 4 && cell_offset_f32(x, q[k], f.h[k], f.h_lo[k], f.c0[k], f.c0_lo[k], &o);
        off[k] = (T)o;
        if (__any_sync(__activemask(), !done)) {
            // (one rounding beside that of x - lo: the centre is not rounded)
            if (!done) off[k] = to_t<T>(fma(-((double)q[k] + 0.5), geo.h[k], x - geo.lo[k]));
        }
        fo[k] = to_f32(off[k]);
    }
    const uint32_t tq = (uint32_t)q[0] << 3;
    pos4[s] = make4(off[0], off[1], off[2], pack_u32(T(0), tq));
    if constexpr (sizeof(T) == 8) fpos[s] = make_float4(fo[0], fo[1], fo[2], __uint_as_float(tq));
    store_hpos(hpos, s, fo[0], fo[1], fo[2], q[0], ph.df);
    cell_s[s] = c;
    src[s] = i | (out ? 0x80000000u : 0u);
}

}  // namespace

}  // namespace mdpd

using namespace mdpd;

extern "C" int mdpd_density_noalloc(const mdpd_params* p, int64_t n, const double* pos,
                                    double* rho, void* cuda_stream)
{
    std::string why;
    auto bad = [&](int code, const std::string& msg) -> int {
        set_global_error("mdpd_density_noalloc: " + msg);
        return code;
    };
    if (!p) return bad(MDPD_ERR_INVALID_ARG, "params is NULL");
    if (n < 0 || n > NA_MAX_PARTICLES)
        return bad(MDPD_ERR_INVALID_ARG, "n must be in 0.." + std::to_string(NA_MAX_PARTICLES));
    if (n > 0 && (!pos || !rho)) return bad(MDPD_ERR_INVALID_ARG, "pos and rho are required");
    if (!(p->rc > 0) || !(p->rd > 0) || !(p->rd <= p->rc) || !std::isfinite(p->rc))
        return bad(MDPD_ERR_INVALID_ARG, "need 0 < rd <= rc");
    if (p->precision != 0 && p->precision != 1)
        return bad(MDPD_ERR_INVALID_ARG, "precision must be 0 or 1");
    Geo geo{};
    geo.ncell = 1;
    for (int k = 0; k < 3; ++k) {
        if (!(p->box[k] > 0) || !std::isfinite(p->box[k]) || !std::isfinite(p->box_lo[k]))
            return bad(MDPD_ERR_INVALID_ARG, "box lengths must be finite and > 0");
        if (p->periodic[k] && p->box[k] < 3.0 * p->rc)
            return bad(MDPD_ERR_INVALID_ARG, "a periodic axis must be at least 3 rc long");
        int m = (int)std::floor(p->box[k] / p->rc);
        if (m < 1) m = 1;
        geo.nc[k] = m;
        geo.periodic[k] = p->periodic[k] ? 1 : 0;
        geo.lo[k] = p->box_lo[k];
        geo.L[k] = p->box[k];
        geo.hi[k] = p->box_lo[k] + p->box[k];
        geo.key_lo[k] = f64_key(geo.lo[k]);
        geo.key_hi[k] = f64_key(geo.hi[k]);
        geo.key_in[k] = f64_key(inside_bound(geo.lo[k], geo.hi[k]));
        geo.h[k] = p->box[k] / m;
        geo.inv_h[k] = 1.0 / geo.h[k];
        geo.ncell *= m;
        if (geo.ncell > NA_MAX_CELLS)
            return bad(MDPD_ERR_INVALID_ARG,
                       "box has more than " + std::to_string(NA_MAX_CELLS) + " cells of edge rc");
    }
    Phys ph{};
    ph.rc = p->rc;
    ph.rd = p->rd;
    ph.rho_self = p->rho_self ? 1 : 0;
    fill_derived(ph, geo);
    cudaStream_t st = (cudaStream_t)cuda_stream;
    // an error left by earlier, unrelated work is not this call's: report it
    // without clearing it
    cudaError_t e = cudaPeekAtLastError();
    if (e != cudaSuccess)
        return bad(MDPD_ERR_CUDA, std::string("a CUDA error was pending before the call: ") +
                                      cudaGetErrorString(e));
    void* base = nullptr;
    int rc = scratch_address(st, &base, why);
    if (rc) return bad(rc, why);
    if (n == 0) return MDPD_OK;

    unsigned char* b = (unsigned char*)base;
    uint32_t* count = (uint32_t*)(b + OFF_COUNT);
    uint32_t* sums = (uint32_t*)(b + OFF_SUMS);
    uint32_t* start = (uint32_t*)(b + OFF_START);
    uint32_t* cellof = (uint32_t*)(b + OFF_CELLOF);
    uint32_t* slot = (uint32_t*)(b + OFF_SLOT);
    uint32_t* key = (uint32_t*)(b + OFF_KEY);
    uint32_t* src = (uint32_t*)(b + OFF_SRC);
    uint32_t* cells = (uint32_t*)(b + OFF_CELLS);
    void* pos4 = b + OFF_POS4;
    float4* fpos = (float4*)(b + OFF_FPOS);
    uint16_t* hpos = (uint16_t*)(b + OFF_HPOS);
    const int nn = (int)n;
    const unsigned nb = (unsigned)((n + 255) / 256);
    // the first failing step names itself (launch errors are this call's own,
    // so they are cleared after being read)
    auto check = [&](const char* what) -> int {
        const cudaError_t le = cudaPeekAtLastError();
        if (le == cudaSuccess) return MDPD_OK;
        cudaGetLastError();
        return bad(MDPD_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(le));
    };
    // counts and tile sums (the launches after the first overlap their predecessors'
    // ends: one shared-memory split for all, see LaunchScope)
    LaunchScope scope(60);
    e = cudaMemsetAsync(count, 0, OFF_START - OFF_COUNT, st);
    if (e != cudaSuccess) return bad(MDPD_ERR_CUDA, std::string("cudaMemsetAsync: ") + cudaGetErrorString(e));
    k_na_count<<<nb, 256, 0, st>>>(nn, pos, geo, ph, cellof, slot, count, sums);
    if ((rc = check("k_na_count"))) return rc;
    launch_scan_from_sums(st, count, geo.ncell, start, sums, nullptr);
    if ((rc = check("cell-count scan"))) return rc;
    launch_pdl(k_na_scatter, dim3(nb), dim3(256), st, nn, cellof, slot, start, key);
    if ((rc = check("k_na_scatter"))) return rc;
    if (p->precision == 0)
        launch_pdl(k_na_gather<double>, dim3(nb), dim3(256), st, nn, pos, key, cellof, start, geo, ph,
                   (D4*)pos4, fpos, hpos, cells, src);
    else
        launch_pdl(k_na_gather<float>, dim3(nb), dim3(256), st, nn, pos, key, cellof, start, geo, ph,
                   (float4*)pos4, fpos, hpos, cells, src);
    if ((rc = check("k_na_gather"))) return rc;
    launch_density_only(st, p->precision, nn, geo, ph, pos4, fpos, hpos, cells, start, src, rho);
    return check("density pass");
}
