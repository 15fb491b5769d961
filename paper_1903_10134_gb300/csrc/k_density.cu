// Density pass that also records each mobile particle's force partners
// (arXiv:1903.10134, Sec. 2.1, Algorithm 1 step 4).
//
// Why lists: in a one-thread-per-particle scan of the 27 neighbour cells only
// about 15 % of the candidates lie within r_c, so a force pass scanning cells
// would execute the ~100 operations of a pair force for nearly every
// candidate with most lanes idle.  The density pass already computes every
// candidate distance; it records the candidates within r_c, and the force
// pass (k_force.cu) runs the pair force only for real partners.  A list entry
// is (j << 5) | image code, where the code (0..26) names the neighbour cell
// offset (ox, oy, oz) that fixes the periodic image of j; so j < 2^27.
// Lists are slot-major (nl[k * cap + column]) so consecutive particles store
// consecutive words; the column is the particle's slot, or, under
// ph.list_compact (frozen-split pass), its block's first slot plus its place
// among the block's mobile particles.  Particles with more than NL_MAX
// partners keep only the count, and the force pass scans their cells
// directly.
#include <cuda_fp16.h>

#include "pair.cuh"

namespace mdpd {

namespace {

// A scaled density term (at most 2^31 in FP32, 2^50 in FP64) rounded to the
// nearest integer, and a fixed-point sum back in the pair precision.
__device__ __forceinline__ unsigned long long to_fixed(float v)
{
    return (unsigned long long)__float2uint_rn(v);
}
__device__ __forceinline__ unsigned long long to_fixed(double v) { return __double2ull_rn(v); }
__device__ __forceinline__ float from_fixed(unsigned long long a, float inv)
{
    const float hi = __uint2float_rn((uint32_t)(a >> 32));
    const float lo = __uint2float_rn((uint32_t)a);
    return fmaf(hi, 4294967296.0f, lo) * inv;
}
__device__ __forceinline__ double from_fixed(unsigned long long a, double inv)
{
    return __ull2double_rn(a) * inv;
}

__device__ __forceinline__ float as_f32(float x) { return x; }
__device__ __forceinline__ float as_f32(double x) { return to_f32(x); }

// Densities of the frozen particles under the frozen split (see
// density_home): rho = frozen-frozen part + the mobile homes' scattered
// terms (and no wall density).
template <typename T>
__global__ void __launch_bounds__(PAIR_BLOCK)
k_frozen_rho(int n, Phys ph, const uint32_t* __restrict__ id_s, const T* __restrict__ rho_ff,
             unsigned long long* __restrict__ facc, T* __restrict__ rho_out)
{
    pdl_enter();
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const T f = rho_ff[id_s[s]];
    if (f < T(0)) return;                       // a mobile particle
    const unsigned long long a = facc[s];
    rho_out[s] = f + from_fixed(a, derived<T>(ph).fix_inv);
    if (a) facc[s] = 0ull;
    if (ph.phi_out != nullptr) ((T*)ph.phi_out)[s] = T(0);
}

// The frozen-frozen part of every frozen particle's density (the sum over its
// frozen neighbours) into rho_ff[id], -1 for mobile ids; one thread per particle
// scanning its 27 neighbour cells.  Runs once per set of wall positions.
// (Candidates are taken by type, so it does not depend on the frozen types the
// binning ordered by.)
template <typename T>
__global__ void __launch_bounds__(PAIR_BLOCK)
k_frozen_part(int n, int64_t cap, Geo geo, Phys ph, const typename Vec4<T>::type* __restrict__ pos4,
              const uint32_t* __restrict__ cell_s, const uint32_t* __restrict__ start,
              const uint32_t* __restrict__ id_s, T* __restrict__ rho_ff)
{
    pdl_enter();
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const Derived<T>& dc = derived<T>(ph);
    const auto pi = pos4[s];
    if (((ph.frozen >> type_of(pi.w)) & 1u) == 0u) {
        rho_ff[id_s[s]] = T(-1);
        return;
    }
    int q0, q1, q2;
    cell_coords(cell_s[s], geo, q0, q1, q2);
    T acc = ph.rho_self ? dc.cw_rho : T(0);
    for (int oz = -1; oz <= 1; ++oz) {
        const int z = neighbour_index(q2, oz, geo.nc[2], geo.periodic[2]);
        if (z < 0) continue;
        const T sz = pi.z - (T)oz * dc.h[2];
        for (int oy = -1; oy <= 1; ++oy) {
            const int y = neighbour_index(q1, oy, geo.nc[1], geo.periodic[1]);
            if (y < 0) continue;
            const T sy = pi.y - (T)oy * dc.h[1];
            for (int ox = -1; ox <= 1; ++ox) {
                const int x = neighbour_index(q0, ox, geo.nc[0], geo.periodic[0]);
                if (x < 0) continue;
                const T sx = pi.x - (T)ox * dc.h[0];
                const uint32_t nc = (uint32_t)(x + geo.nc[0] * (y + geo.nc[1] * z));
                uint32_t b = start[nc], e = start[nc + 1];
                if (!MDPD_DBG_OK(b <= e && e <= (uint32_t)cap, ph.dbg_status)) e = b;
                for (uint32_t j = b; j < e; ++j) {
                    const auto pj = pos4[j];
                    const T dx = sx - pj.x, dy = sy - pj.y, dz = sz - pj.z;
                    const T r2 = dx * dx + dy * dy + dz * dz;
                    if (r2 < dc.rc2 && ((ph.frozen >> type_of(pj.w)) & 1u) && j != (uint32_t)s) {
                        const T w = max(T(1) - sqrt_fast(r2) * dc.inv_rd, T(0));
                        const T term = dc.cw_rho * w * w;      // r = 0 gives w(0)
                        acc += term;
                    }
                }
            }
        }
    }
    rho_ff[id_s[s]] = acc;
}

// One thread per home particle, in two phases.
//   1. A filter over the candidates of the 27 neighbour cells: the cells of a row
//      (fixed y and z) are consecutive in slot order, so a home scans nine runs of
//      three cells (two runs in a row cut by a periodic face), and of every
//      candidate only the sign of r^2 - (1 + margin) is kept, shifted into a bit
//      mask: no branch.  It runs on FP16 positions in units of r_c (hpos), two
//      candidates an instruction, four a load; FILT covers their rounding, so a
//      partner is never lost.
//   2. The set bits in candidate order: the separation from the cell offsets in the
//      pair precision, the exact test, the density term, the list entry.
// Doing all of it per candidate kept 14 of 32 lanes busy on the rock: the hits (one
// candidate in seven, in different lanes at different times) ran their thirty
// instructions for nearly every candidate of the warp.  Here a warp meets them
// about 31 times instead of 163.
//
// Runs and masks wait in shared memory, in one array: the masks of the runs done
// (empty ones skipped) take the places of those runs.  A home with more masks than
// that (runs longer than 32 candidates) works them off and goes on.
//
// The rows are taken in the order of dn_row, in four groups: the home's own, with ten of
// the 25 hits, then three, two and three of the others, with two, six and seven.  In
// systems of few particles (density_groups), where one lane's chain of 5,000 instructions
// is the pass's time, LPH = 4 lanes share a home and take one group each.  The first
// writes its hits to the list; those of the others wait in shared memory, each lane's
// behind the filter's count of those before it, and follow it; the density is the sum of
// the groups' in their order.  A home whose hits do not fit counts them first and finds
// them again for the list.  In a batch a replica's home may have one lane where its
// system alone has four: the lane then sums the groups apart as well (ph.rho_groups,
// fold), so that the replica stays that system to the bit.
__device__ constexpr int dn_row(int k) { return (int)(0x75318624ull >> 4 * k & 15u); }
constexpr uint32_t DN_GROUP = 0x1dc9bu;       // group of a row, two bits each
constexpr int DN_POOL = 45;        // hits kept for a home (LPH > 1); odd, for the banks
// r^2 < FILT passes (1 + 9 * 2^-10, exact in FP16).  With u = 2^-10 an |x| < 4 is off by
// u at most, home and candidate; |y|, |z| < 1 of a candidate by u / 4, < 3 of a home
// by u; a difference near 1 by u / 2 more.  That is 2.5 u in x and 1.75 u in y and z,
// 3.5 u in the separation and 7.1 u in r^2 near 1, and the three squares' sums add
// u / 2: below 8 u.
constexpr float FILT = 1.0f + 9.0f / 1024.0f;

template <typename T, int LPH>
struct DensitySmem {
    static constexpr int ROWS = LPH == 1 ? 9 : 3;     // of a lane, at most
    static constexpr int RUNS = 2 * ROWS;
    // FP64: candidates near r_d kept before they are evaluated
    static constexpr int NEAR = sizeof(T) == 4 ? 1 : LPH == 1 ? 32 : 16;
    // run: length, first slot | across a face in x << 27 | row << 28
    // mask: candidates from the top bit, first slot | across << 27 | row << 28
    uint32_t a[RUNS][PAIR_BLOCK];
    uint32_t b[RUNS][PAIR_BLOCK];
    typename Vec4<T>::type shift[27];          // image shift of a neighbour-cell code
    float4 fshift[sizeof(T) == 8 ? 27 : 1];    // the same in FP32
    uint32_t near[NEAR][sizeof(T) == 4 ? 1 : PAIR_BLOCK];
    uint32_t hit[LPH == 1 ? 1 : PAIR_BLOCK / LPH][DN_POOL];
};

// Density terms and sums with each operation rounded, so that the two ways of
// adding them (LPH) agree.
__device__ __forceinline__ float rho_term(float cw, float w) { return __fmul_rn(__fmul_rn(cw, w), w); }
__device__ __forceinline__ double rho_term(double cw, double w) { return __dmul_rn(__dmul_rn(cw, w), w); }
__device__ __forceinline__ float rho_add(float a, float t) { return __fadd_rn(a, t); }
__device__ __forceinline__ double rho_add(double a, double t) { return __dadd_rn(a, t); }

// k as a float for k < 2^23 (the conversion instruction runs at an eighth of the rate)
__device__ __forceinline__ float small_float(uint32_t k)
{
    return __uint_as_float(0x4b000000u | k) - 8388608.0f;
}

// (t < 0) of four FP16 numbers, in order, into m from the right.
__device__ __forceinline__ uint32_t push_signs(uint32_t m, __half2 t01, __half2 t23)
{
    const uint32_t u = *reinterpret_cast<const uint32_t*>(&t01),
                   v = *reinterpret_cast<const uint32_t*>(&t23);
    m = __funnelshift_l(u << 16, m, 1);
    m = __funnelshift_l(u, m, 1);
    m = __funnelshift_l(v << 16, m, 1);
    return __funnelshift_l(v, m, 1);
}
__device__ __forceinline__ __half2 as_half2(uint32_t u) { return *reinterpret_cast<__half2*>(&u); }

template <typename T, int LPH>
__device__ __forceinline__ void fill_shift(DensitySmem<T, LPH>& sm, const Phys& ph)
{
    const int c = threadIdx.x;
    if (c >= 27) return;
    const Derived<T>& dc = derived<T>(ph);
    sm.shift[c] = make4((T)(c % 3 - 1) * dc.h[0], (T)((c / 3) % 3 - 1) * dc.h[1],
                        (T)(c / 9 - 1) * dc.h[2], T(0));
    if constexpr (sizeof(T) == 8)
        sm.fshift[c] = make_float4((float)(c % 3 - 1) * ph.df.h[0], (float)((c / 3) % 3 - 1) * ph.df.h[1],
                                   (float)(c / 9 - 1) * ph.df.h[2], 0.0f);
}

// The density and partner list of the home in slot s; column lcol of the list.
// With LPH > 1 the LPH lanes of a group call it together.
template <typename T, bool WANT_PHI, int FS, int LPH, bool FOLD>
__device__ __forceinline__ void density_home(
    DensitySmem<T, LPH>& sm, int s, int64_t cap, const Geo& geo, const Phys& ph, int64_t cell0,
    const typename Vec4<T>::type* __restrict__ pos4, const float4* __restrict__ fpos,
    const uint4* __restrict__ hpos, const uint32_t* __restrict__ cell_s,
    const uint32_t* __restrict__ start, T* __restrict__ rho_out, uint32_t* __restrict__ nl,
    uint32_t* __restrict__ nl_count, unsigned long long* __restrict__ facc, int64_t lcol,
    const uint32_t* __restrict__ src = nullptr, double* __restrict__ out = nullptr)
{
    static_assert(LPH == 1 || LPH == 4, "lanes per home");
    constexpr bool LIST = FS != 3;
    const Derived<T>& dc = derived<T>(ph);
    const Derived<float>& df = ph.df;
    const int tid = threadIdx.x;
    const int sub = LPH == 1 ? 0 : tid % LPH;
    const unsigned group = LPH == 1 ? 0u : ((1u << LPH) - 1u) << ((tid & 31) & ~(LPH - 1));
    const auto pi = pos4[s];
    int q0, q1, q2;
    cell_coords(cell_s[s], geo, q0, q1, q2);

    // the runs: rows (oy, oz) in order, the part across the lower face in x first,
    // the part across the upper one last
    const bool lo_x = geo.periodic[0] && q0 == 0, hi_x = geo.periodic[0] && q0 == geo.nc[0] - 1;
    const int xb0 = max(q0 - 1, 0), xe0 = min(q0 + 1, geo.nc[0] - 1) + 1;
    constexpr int ROWS = DensitySmem<T, LPH>::ROWS;
    constexpr uint32_t SPLIT = LPH == 1 ? 0x90u : 0x96410u;
    const int k0 = (int)(SPLIT >> 4 * sub & 15u), kend = (int)(SPLIT >> 4 * (sub + 1) & 15u);
    int nrun = 0;
    auto build_runs = [&]() {
        uint32_t b[ROWS], e[ROWS];
        auto row_start = [&](int k) -> const uint32_t* {
            const int r = dn_row(k), oz = r * 11 >> 5;
            const int z = neighbour_index(q2, oz - 1, geo.nc[2], geo.periodic[2]);
            const int y = neighbour_index(q1, r - 3 * oz - 1, geo.nc[1], geo.periodic[1]);
            return k < kend && z >= 0 && y >= 0 ? start + cell0 + geo.nc[0] * (y + geo.nc[1] * z)
                                                : nullptr;
        };
#pragma unroll
        for (int k = 0; k < ROWS; ++k) {
            const uint32_t* st = row_start(k0 + k);
            b[k] = st ? st[xb0] : 0u;
            e[k] = st ? st[xe0] : 0u;
        }
        nrun = 0;
        auto put = [&](uint32_t first, uint32_t end, uint32_t code) {
            if (first < end && MDPD_DBG_OK(end <= (uint32_t)cap, ph.dbg_status)) {
                sm.a[nrun][tid] = end - first;
                sm.b[nrun][tid] = first | code << 27;
                ++nrun;
            }
        };
#pragma unroll
        for (int k = 0; k < ROWS; ++k) {
            const uint32_t r = (uint32_t)dn_row(k0 + k);
            if (lo_x || hi_x) {
                const uint32_t* st = row_start(k0 + k);
                if (!st) continue;
                const int x = lo_x ? geo.nc[0] - 1 : 0;
                if (hi_x) put(b[k], e[k], r << 1);
                put(st[x], st[x + 1], r << 1 | 1u);
                if (lo_x) put(b[k], e[k], r << 1);
            } else {
                put(b[k], e[k], r << 1);
            }
        }
    };
    const bool mob_true = ((ph.frozen >> type_of(pi.w)) & 1u) == 0u;
    const bool mobile = LIST && (ph.list_all || mob_true);
    // wall density of a mobile particle (WANT_PHI): sum over frozen partners
    // within r_c of 15/(2 pi r_c^3) (1 - r/r_c)^2
    const bool want_phi = WANT_PHI && mob_true;
    T acc = ph.rho_self ? dc.cw_rho : T(0), phi = T(0);
    // part: the sum of the current group of rows, which fold adds to acc
    T part = acc;
    acc = T(0);
    if (LPH > 1 && sub != 0) part = T(0);
    uint32_t group_now = 0;
    auto fold = [&](uint32_t jr) {
        const uint32_t g = (DN_GROUP >> 2 * (jr >> 28)) & 3u;
        if (g == group_now) return;
        acc = rho_add(acc, part);
        part = T(0);
        group_now = g;
    };
    uint32_t cnt = 0;
    uint32_t* lp = nl + lcol;                   // next list entry: nl[cnt * cap + lcol]
    // cell column of a candidate across a periodic face, from the home's
    const int across = q0 == 0 ? -geo.nc[0] : geo.nc[0];
    // the home in FP16, in units of r_c: x in the window of four cells that holds the
    // columns q0 - 1 .. q0 + 1
    const float ox = as_f32(pi.x), oy = as_f32(pi.y), oz = as_f32(pi.z);
    const float hn1 = df.h[1] * df.inv_rc, hn2 = df.h[2] * df.inv_rc;
    const float oy1 = oy * df.inv_rc, oz1 = oz * df.inv_rc;
    const bool win_b = ((q0 + 1) & 3) < 2;
    auto x_in_window = [&](int col, int off) {
        return __float2half2_rn(fmaf((float)(2 * ((col & 3) + off) - 3), 0.5f * df.h[0], ox) * df.inv_rc);
    };
    const __half2 hx0 = x_in_window(q0 + (win_b ? 2 : 0), 0);
    const __half2 thr = __float2half2_rn(-FILT);
    __half2 hx = hx0, hy = hx0, hz = hx0;
    bool xb = win_b;

    // pass 0: every lane its rows (LPH > 1: hits kept, or counted if they do not fit);
    // pass 1, if they did not: once more for the list
    uint32_t nhit = 0, pool = 0;
    bool fits = true;
    for (int pass = 0; pass < (LPH == 1 ? 1 : 2); ++pass) {
    if (LPH > 1 && pass == 1 && sub == 0) break;
    build_runs();
    // place of mask k: the runs' done ones, before them (LPH > 1) the never used ones
    auto place = [&](int k) {
        if (LPH == 1) return k;
        const int q = nrun + k;
        return q >= DensitySmem<T, LPH>::RUNS ? q - DensitySmem<T, LPH>::RUNS : q;
    };
    int run = 0;
    uint32_t len = 0, rb = 0;
    for (bool first = LPH > 1 && pass == 0; first || run < nrun || len; first = false) {
        int nw = 0;
        uint32_t npass = 0;
        while (run < nrun || len) {
            uint32_t lead = 0;
            if (len == 0) {
                len = sm.a[run][tid];
                rb = sm.b[run][tid];
                ++run;
                const int r = (int)(rb >> 28), rz = (r * 11) >> 5, ry = r - 3 * rz;
                hy = __float2half2_rn(fmaf(small_float((uint32_t)ry) - 1.0f, -hn1, oy1));
                hz = __float2half2_rn(fmaf(small_float((uint32_t)rz) - 1.0f, -hn2, oz1));
                hx = hx0;
                xb = win_b;
                if (rb & 1u << 27) {
                    // across a periodic face: one cell, met from the column beside it
                    hx = q0 == 0 ? x_in_window(geo.nc[0] - 1, 1) : x_in_window(0, -1);
                    xb = false;
                }
                // whole groups of four slots: the candidates before the run's are
                // dropped from the mask
                lead = rb & 3u;
                rb -= lead;
                len += lead;
            }
            const uint32_t k1 = min(len, 32u);
            const uint4* f = hpos + (size_t)((rb & 0x07ffffffu) >> 2) * 2;
            uint32_t m = 0;
#pragma unroll 2
            for (uint32_t k = 0; k < k1; k += 4, f += 2) {
                const uint4 yz = f[0];
                const uint2 x = reinterpret_cast<const uint2*>(f + 1)[xb];
                const __half2 dx0 = hx - as_half2(x.x), dx1 = hx - as_half2(x.y);
                const __half2 dy0 = hy - as_half2(yz.x), dy1 = hy - as_half2(yz.y);
                const __half2 dz0 = hz - as_half2(yz.z), dz1 = hz - as_half2(yz.w);
                m = push_signs(m, __hfma2(dz0, dz0, __hfma2(dy0, dy0, __hfma2(dx0, dx0, thr))),
                               __hfma2(dz1, dz1, __hfma2(dy1, dy1, __hfma2(dx1, dx1, thr))));
            }
            m = (m >> ((0u - k1) & 3u)) << (32u - k1) & (0xffffffffu >> lead);
            // not the home itself: its own term is left out of the sum rather than
            // taken off it (it is the largest, and the sum's rounding would grow)
            const uint32_t self = (uint32_t)s - (rb & 0x07ffffffu);
            if (self < 32u) m &= ~(0x80000000u >> self);
            if (m) {
                sm.a[place(nw)][tid] = m;
                sm.b[place(nw)][tid] = rb;
                ++nw;
                if (LPH > 1) npass += (uint32_t)__popc(m);
            }
            rb += k1;
            len -= k1;
            // no place free until masks are worked off
            if (nw == run + (LPH > 1 ? DensitySmem<T, LPH>::RUNS - nrun : 0) && len) break;
        }
        if (LPH > 1 && first) {
            uint32_t all = 0;
#pragma unroll
            for (int t = 0; t < LPH; ++t) {
                const uint32_t nt = t == 0 ? 0u : __shfl_sync(group, npass, t, LPH);
                pool += t < sub ? nt : 0u;
                all += nt;
            }
            fits = __all_sync(group, all <= (uint32_t)DN_POOL &&
                                         (sub == 0 || (run == nrun && len == 0u)));
        }
        if (nw == 0) break;

        // the set bits, one ahead of the one worked on
        int w = 0;
        uint32_t m = sm.a[place(0)][tid], base = sm.b[place(0)][tid];
        uint32_t j1 = 0;
        auto next = [&]() {
            const int b = __clz((int)m);
            j1 = base + (uint32_t)b;           // row and face bits above the slot
            m ^= 0x80000000u >> b;
            if (m == 0u && ++w < nw) {
                m = sm.a[place(w)][tid];
                base = sm.b[place(w)][tid];
            }
        };
        // neighbour-cell code of a candidate in cell column qj, jr as from next()
        auto code_of = [&](uint32_t qj, uint32_t jr) {
            const int ox = (int)qj - q0 + (jr & 1u << 27 ? across : 0);
            return 3 * (int)(jr >> 28) + ox + 1;
        };
        auto append = [&](uint32_t j, int code) {
            const uint32_t entry = j << 5 | (uint32_t)code;   // (bits above the slot shift out)
            if (LPH > 1 && pass == 0 && sub != 0) {
                if (fits) sm.hit[tid / LPH][pool + nhit] = entry;
                ++nhit;
                return;
            }
            if (cnt < (uint32_t)NL_MAX) *lp = entry;
            lp += cap;
            ++cnt;
        };
        next();
        if constexpr (sizeof(T) == 4) {
            float4 p1 = pos4[j1 & 0x07ffffffu];
            for (;;) {
                const uint32_t jr = j1;
                const float4 pj = p1;
                const bool more = w < nw;
                if (more) {
                    next();
                    p1 = pos4[j1 & 0x07ffffffu];
                }
                const uint32_t bits = __float_as_uint(pj.w);
                const int code = code_of(bits >> 3, jr);
                const float4 sh = sm.shift[code];
                const float dx = pi.x - sh.x - pj.x, dy = pi.y - sh.y - pj.y,
                            dz = pi.z - sh.z - pj.z;
                const float r2 = dx * dx + dy * dy + dz * dz;
                if (r2 < dc.rc2) {
                    const float wr = max(1.0f - sqrt_fast(r2) * dc.inv_rd, 0.0f);
                    const float term = rho_term(dc.cw_rho, wr);  // r = 0 gives w(0)
                    if (pass == 0) {
                        if (FOLD && ph.rho_groups) fold(jr);
                        part = rho_add(part, term);
                    }
                    const bool fz = (FS == 1 || WANT_PHI) && ((ph.frozen >> (bits & 7u)) & 1u);
                    if (FS == 1 && fz && term > 0.0f && pass == 0)
                        atomicAdd(facc + (jr & 0x07ffffffu), to_fixed(term * dc.fix_scale));
                    if (mobile && r2 > 0.0f) {      // not coincident
                        append(jr, code);
                        if (want_phi && fz && pass == 0) {
                            const float wq = 1.0f - sqrt_t(r2) * dc.inv_rc;
                            phi += dc.cw_phi * wq * wq;
                        }
                    }
                }
                if (!more) break;
            }
        } else {
            // FP64 arithmetic runs at 1/64 of the FP32 rate: the FP32 distance
            // (error below 2e-6 r_c^2) decides all but the pairs within 1e-5 of the
            // cutoff, and only those near or within r_d are evaluated in FP64, in a
            // loop of their own
            const float rc2 = df.rc2, eps = 1e-5f * rc2, near2 = df.rd2 + eps;
            int nnear = 0;
            auto r2_of = [&](uint32_t j, int code) {
                const auto pj = pos4[j];
                const auto sh = sm.shift[code];
                const T dx = pi.x - sh.x - pj.x, dy = pi.y - sh.y - pj.y, dz = pi.z - sh.z - pj.z;
                return dx * dx + dy * dy + dz * dz;
            };
            auto evaluate = [&](uint32_t entry) {
                const uint32_t j = entry >> 5;
                const T r2 = r2_of(j, (int)(entry & 31u));
                if (r2 < dc.rc2) {
                    if (FOLD && ph.rho_groups) fold((entry & 31u) * 11u >> 5 << 28);
                    const T wr = max(T(1) - sqrt_fast(r2) * dc.inv_rd, T(0));
                    const T term = rho_term(dc.cw_rho, wr);      // r = 0 gives w(0)
                    part = rho_add(part, term);
                    const bool fz = (FS == 1 || WANT_PHI) &&
                                    ((ph.frozen >> type_of(pos4[j].w)) & 1u);
                    if (FS == 1 && fz && term > T(0))
                        atomicAdd(facc + j, to_fixed(term * dc.fix_scale));
                    if (want_phi && fz && r2 > T(0)) {
                        const T wq = T(1) - sqrt_t(r2) * dc.inv_rc;
                        phi += dc.cw_phi * wq * wq;
                    }
                }
            };
            auto evaluate_near = [&]() {
                for (int k = 0; k < nnear; ++k) evaluate(sm.near[k][tid]);
                nnear = 0;
            };
            float4 p1 = fpos[j1 & 0x07ffffffu];
            for (;;) {
                const uint32_t jr = j1;
                const float4 pj = p1;
                const bool more = w < nw;
                if (more) {
                    next();
                    p1 = fpos[j1 & 0x07ffffffu];
                }
                const uint32_t bits = __float_as_uint(pj.w);
                const int code = code_of(bits >> 3, jr);
                const float4 sh = sm.fshift[code];
                const float dx = ox - sh.x - pj.x, dy = oy - sh.y - pj.y, dz = oz - sh.z - pj.z;
                const float r2 = dx * dx + dy * dy + dz * dz;
                const uint32_t entry = jr << 5 | (uint32_t)code;
                // (a NaN takes the exact path)
                bool in = true;
                if (!(r2 < rc2 - eps) || !(r2 > eps)) {
                    const T q = r2_of(entry >> 5, code);
                    in = q < dc.rc2 && q > T(0);
                }
                if (mobile && in) append(jr, code);
                if (pass == 0 && (!(r2 >= near2) || (want_phi && ((ph.frozen >> (bits & 7u)) & 1u)))) {
                    sm.near[nnear++][tid] = entry;
                    if (nnear == DensitySmem<T, LPH>::NEAR) evaluate_near();
                }
                if (!more) break;
            }
            evaluate_near();
        }
    }
    if constexpr (LPH > 1) {
        if (pass == 1) break;
        uint32_t all = 0, before = 0;
        T sum = T(0);
#pragma unroll
        for (int t = 0; t < LPH; ++t) {
            const uint32_t ht = __shfl_sync(group, sub == 0 ? cnt : nhit, t, LPH);
            sum = rho_add(sum, __shfl_sync(group, part, t, LPH));
            before += t < sub ? ht : 0u;
            all += ht;
        }
        acc = sum;
        // wall density: the lanes' sums in a fixed order
        if (WANT_PHI)
#pragma unroll
            for (int o = 1; o < LPH; o <<= 1) phi += __shfl_xor_sync(group, phi, o);
        if (LIST && fits)
            for (uint32_t k = 0; k < nhit; ++k)
                if (before + k < (uint32_t)NL_MAX)
                    lp[(int64_t)(before + k) * cap] = sm.hit[tid / LPH][pool + k];
        if (sub != 0) {
            cnt = before;
            lp += (int64_t)before * cap;
        }
        pool = all;                            // the home's hits
        if (!LIST || fits || all == 0u) break;
    }
    }
    if constexpr (LPH > 1) {
        cnt = pool;
        __syncwarp(group);                     // the pool is read before the next home's
    } else {
        acc = rho_add(acc, part);
    }
    if (sub != 0) return;
    if constexpr (!LIST) {
        const uint32_t f = src[s], i = f & 0x7fffffffu;
        if ((int64_t)i < cap) out[i] = f >> 31 ? __longlong_as_double(0x7ff8000000000000ll) : (double)acc;
        return;
    }
    rho_out[s] = acc;
    nl_count[s] = cnt;
    if (WANT_PHI) ((T*)ph.phi_out)[s] = phi;
}

// Frozen split (FS, single systems with frozen particles, under
// MDPD_KERNELS_NLIST_THREAD or with the wall density; the rule and its timings are at
// engine.cu: splits).  Frozen particles never move, so the part of a frozen particle's
// density that comes from frozen neighbours is a constant, computed once
// (k_frozen_part).  FS = 1 then scans for mobile homes only: a mobile home adds each
// frozen candidate's share w_rho(r_ij) of that candidate's density (the same term it
// adds to its own) to facc[j] as a fixed-point integer (Derived::fix_scale), by atomic
// addition, so the sum does not depend on the order; k_frozen_rho then forms
// rho_j = rho_ff + facc * fix_inv and clears facc.  Each FS = 1 block gathers
// the mobile homes of R * PAIR_BLOCK slots (R = frozen_rounds) and runs them in
// rounds, so no warp is spent on frozen homes.  FS = 3: densities only, to out[src[s]]
// (NaN where src has its top bit set).  FS = 0: every particle is
// a home, and partner lists are written for mobile ones (all under list_all).
//
// Bound by issue (77 % of the cycles on the rock of 256^3 voxels, L1 data path 58 %): per
// 32 homes of a slab 376 instructions for the runs, 2,228 in the filter, 2,421 for the
// hits.  Density pass in FP32 before (each candidate in full by one thread, or a warp per
// cell) and with the filter, us: slab of 820,000 219 / 141, rock of 256^3 voxels (frozen
// split) 776 / 480, batch of 256 liquids (2.8 million) 710 / 476; small systems at
// density_groups.
template <typename T, bool BATCH, bool WANT_PHI, int FS, int LPH, int R>
__global__ void __launch_bounds__(PAIR_BLOCK, sizeof(T) == 4 ? 8 : 5)
k_density_nl(int n, int64_t cap, Geo geo_p, Phys ph_p, Batch bt,
             const typename Vec4<T>::type* __restrict__ pos4, const float4* __restrict__ fpos,
             const uint4* __restrict__ hpos, const uint32_t* __restrict__ cell_s,
             const uint32_t* __restrict__ start, T* __restrict__ rho_out,
             uint32_t* __restrict__ nl, uint32_t* __restrict__ nl_count,
             unsigned long long* __restrict__ facc, const uint32_t* __restrict__ src,
             double* __restrict__ out)
{
    static_assert(FS == 0 || !BATCH, "the frozen split is for single systems");
    __shared__ DensitySmem<T, LPH> sm;
    constexpr int HOMES = PAIR_BLOCK / LPH;    // homes of a round
    constexpr bool FOLD = BATCH && LPH == 1;
    pdl_enter();
    if constexpr (FS == 1) {
        // the mobile homes of R * PAIR_BLOCK slots, in slot order (LPH blocks share
        // them: each takes HOMES of every PAIR_BLOCK)
        __shared__ int act[R * PAIR_BLOCK];
        __shared__ uint32_t wcnt[R][PAIR_BLOCK / 32];
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const unsigned lt = (1u << lane) - 1u;
        const int64_t base = (int64_t)(blockIdx.x / LPH) * (R * PAIR_BLOCK);
        fill_shift(sm, ph_p);
        unsigned bm[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int64_t t = base + r * PAIR_BLOCK + threadIdx.x;
            const bool mob = t < n && ((ph_p.frozen >> type_of(pos4[t].w)) & 1u) == 0u;
            bm[r] = __ballot_sync(0xffffffffu, mob);
            if (lane == 0) wcnt[r][warp] = (uint32_t)__popc(bm[r]);
        }
        __syncthreads();
        uint32_t nmob = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            uint32_t off = nmob;
#pragma unroll
            for (int w = 0; w < PAIR_BLOCK / 32; ++w) {
                off += w < warp ? wcnt[r][w] : 0u;
                nmob += wcnt[r][w];
            }
            if ((bm[r] >> lane) & 1u)
                act[off + __popc(bm[r] & lt)] = (int)(base + r * PAIR_BLOCK + threadIdx.x);
        }
        __syncthreads();
        // list column: the home's slot, or (list_compact) the block's first
        // slot plus the home's place among its mobile homes, which the force
        // pass's rounds blocks form the same way (consecutive columns for a
        // warp's homes: coalesced list stores and loads)
        for (uint32_t q = blockIdx.x % LPH * HOMES + threadIdx.x / LPH; q < nmob; q += PAIR_BLOCK)
            density_home<T, WANT_PHI, FS, LPH, false>(sm, act[q], cap, geo_p, ph_p, 0, pos4, fpos, hpos,
                                               cell_s, start, rho_out, nl, nl_count, facc,
                                               ph_p.list_compact ? base + q : (int64_t)act[q]);
        return;
    }
    // a single system: one round of homes per block; a batch: a chunk's slots in rounds
    int first, count;
    int64_t cell0 = 0;
    const Rep* rp = nullptr;
    if constexpr (BATCH) {
        const int4 ch = bt.chunks[blockIdx.x / LPH];
        rp = &block_rep<REP_SCALARS>(bt.reps, ch.x);
        const int part = (int)(blockIdx.x % LPH) * HOMES;
        first = ch.y + part;
        count = min(HOMES, ch.z - part);
        cell0 = rp->cell0;
    } else {
        first = blockIdx.x * HOMES;
        count = min(HOMES, n - first);
    }
    fill_shift(sm, BATCH ? rp->ph : ph_p);
    __syncthreads();
    const int k = (int)threadIdx.x / LPH;
    if (k >= count) return;
    density_home<T, WANT_PHI, FS, LPH, FOLD>(sm, first + k, cap, BATCH ? rp->geo : geo_p,
                                       BATCH ? rp->ph : ph_p, cell0, pos4, fpos, hpos, cell_s, start,
                                       rho_out, nl, nl_count, facc, (int64_t)(first + k), src, out);
}

}  // namespace

template <typename T, int R>
static void density_t(cudaStream_t st, int n, int64_t cap, const Geo& geo, const Phys& ph,
                      const void* pos4, const void* fpos, const uint16_t* hpos,
                      const uint32_t* cell_s, const uint32_t* start, void* rho, uint32_t* nl,
                      uint32_t* nl_count, int fs, unsigned long long* facc, const uint32_t* id_s,
                      void* rho_ff)
{
    using V = typename Vec4<T>::type;
    const int nb = (n + PAIR_BLOCK - 1) / PAIR_BLOCK;
    if (fs == 2) {
        launch_pdl(k_frozen_part<T>, dim3(nb), dim3(PAIR_BLOCK), st, n, cap, geo, ph,
                   (const V*)pos4, cell_s, start, id_s, (T*)rho_ff);
        return;
    }
    const bool phi = ph.phi_out != nullptr;
    const int lph = R == 1 && ph.rho_groups ? 4 : 1;
    auto k = fs == 1 ? (phi ? k_density_nl<T, false, true, 1, 1, R> : k_density_nl<T, false, false, 1, 1, R>)
                     : (phi ? k_density_nl<T, false, true, 0, 1, 1> : k_density_nl<T, false, false, 0, 1, 1>);
    if constexpr (R == 1)
        if (lph == 4)
            k = fs == 1 ? (phi ? k_density_nl<T, false, true, 1, 4, R> : k_density_nl<T, false, false, 1, 4, R>)
                        : (phi ? k_density_nl<T, false, true, 0, 4, 1> : k_density_nl<T, false, false, 0, 4, 1>);
    const int per = (fs == 1 ? R * PAIR_BLOCK : PAIR_BLOCK) / lph;     // slots of a block
    launch_pdl(k, dim3((n + per - 1) / per), dim3(PAIR_BLOCK), st, n, cap, geo, ph, Batch{},
               (const V*)pos4, (const float4*)fpos, (const uint4*)hpos, cell_s, start, (T*)rho, nl,
               nl_count, facc, (const uint32_t*)nullptr, (double*)nullptr);
    if (fs == 1)
        launch_pdl(k_frozen_rho<T>, dim3(nb), dim3(PAIR_BLOCK), st, n, ph, id_s,
                   (const T*)rho_ff, facc, (T*)rho);
}

void launch_density_nl(cudaStream_t st, int precision, int n, int64_t cap, const Geo& geo,
                       const Phys& ph, const void* pos4, const void* fpos, const uint16_t* hpos,
                       const uint32_t* cell_s, const uint32_t* start, void* rho, uint32_t* nl,
                       uint32_t* nl_count, int fs, unsigned long long* facc, const uint32_t* id_s,
                       void* rho_ff)
{
    if (n <= 0) return;
    const bool rounds = frozen_rounds(n) > 1;
    auto f = precision == 0 ? (rounds ? density_t<double, FORCE_ROUNDS> : density_t<double, 1>)
                            : (rounds ? density_t<float, FORCE_ROUNDS> : density_t<float, 1>);
    f(st, n, cap, geo, ph, pos4, fpos, hpos, cell_s, start, rho, nl, nl_count, fs, facc, id_s, rho_ff);
}

template <typename T, int LPH>
static void density_batch_t(cudaStream_t st, int64_t cap, const Batch& bt, const void* pos4,
                            const void* fpos, const uint16_t* hpos, const uint32_t* cell_s,
                            const uint32_t* start, void* rho, uint32_t* nl, uint32_t* nl_count)
{
    launch_pdl_smem(k_density_nl<T, true, false, 0, LPH, 1>, dim3(bt.nchunk * LPH), dim3(PAIR_BLOCK),
                    REP_SMEM, st, 0, cap, Geo{}, Phys{}, bt, (const typename Vec4<T>::type*)pos4,
                    (const float4*)fpos, (const uint4*)hpos, cell_s, start, (T*)rho, nl, nl_count,
                    nullptr, (const uint32_t*)nullptr, (double*)nullptr);
}

void launch_density_only(cudaStream_t st, int precision, int n, const Geo& geo, const Phys& ph,
                         const void* pos4, const void* fpos, const uint16_t* hpos,
                         const uint32_t* cell_s, const uint32_t* start, const uint32_t* src, double* out)
{
    if (n <= 0) return;
    auto go = [&](auto t, auto k, int lph) {
        using T = decltype(t);
        const int per = PAIR_BLOCK / lph;
        launch_pdl(k, dim3((n + per - 1) / per), dim3(PAIR_BLOCK), st, n, (int64_t)n, geo, ph, Batch{},
                   (const typename Vec4<T>::type*)pos4, (const float4*)fpos, (const uint4*)hpos, cell_s,
                   start, (T*)nullptr, (uint32_t*)nullptr, (uint32_t*)nullptr,
                   (unsigned long long*)nullptr, src, out);
    };
    const bool shared = density_groups(precision, n);
    if (precision == 0 && shared) go(double{}, k_density_nl<double, false, false, 3, 4, 1>, 4);
    else if (precision == 0) go(double{}, k_density_nl<double, false, false, 3, 1, 1>, 1);
    else if (shared) go(float{}, k_density_nl<float, false, false, 3, 4, 1>, 4);
    else go(float{}, k_density_nl<float, false, false, 3, 1, 1>, 1);
}

void launch_density_nl_batch(cudaStream_t st, int precision, int64_t cap, const Batch& bt,
                             const void* pos4, const void* fpos, const uint16_t* hpos,
                             const uint32_t* cell_s, const uint32_t* start, void* rho, uint32_t* nl,
                             uint32_t* nl_count)
{
    if (bt.nchunk <= 0) return;
    const bool shared = density_groups(precision, (int64_t)bt.nchunk * PAIR_BLOCK);
    auto f = precision == 0 ? (shared ? density_batch_t<double, 4> : density_batch_t<double, 1>)
                            : (shared ? density_batch_t<float, 4> : density_batch_t<float, 1>);
    f(st, cap, bt, pos4, fpos, hpos, cell_s, start, rho, nl, nl_count);
}

}  // namespace mdpd
