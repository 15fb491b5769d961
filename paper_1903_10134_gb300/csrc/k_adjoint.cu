// Adjoint (vector-Jacobian products) of one mDPD force evaluation and of a
// velocity-Verlet window (Sec. 2.1, Eq. 1 and Algorithm 1 of
// arXiv:1903.10134), for single systems and batches of replicas.
//
// One force evaluation maps (x, u, theta) to a_i = sum_j f_ij (i mobile),
// with rho_i = sum_j w_rho(r_ij) recomputed from x, u the velocities the
// dissipative term sees and theta = (A, B, gamma).  Its conservative virial is
// W_ab = 1/2 sum_{i mobile} sum_j d_a F^C_b.  Given abar (the adjoint of the
// accelerations, id order) and, optionally, weights c of the six virial
// components (per replica), the kernels return the gradient of
//     L = sum_i abar_i . a_i + sum_k c_k W_k
// with respect to positions, to u and to the symmetric tables A, B, gamma,
// the random draws of the step held fixed.
//
// For a pair (i, j): d = x_i - x_j, r = |d|, e = d / r, w = e . u_ij,
//   s   = A wc + B (rho_i + rho_j) wd [r < r_d] - gamma wc^2 w + sigma wc xi / sqrt(dt)
//   s_c = A wc + B (rho_i + rho_j) wd [r < r_d]            (conservative part)
// Force part, q = abar_i - abar_j (frozen particles have no acceleration, so
// their abar counts as zero):
//   xbar_i += (q.e)(s_r e + s_w (u_ij - w e) / r) + s (q - (q.e) e) / r
//   ubar_i += (q.e) s_w e,     rhobar_i += (q.e) B wd [r < r_d]
// (s_r = ds/dr at fixed w and rho, s_w = -gamma wc^2).  Virial part, with the
// quadratic form Q(d) = c_xx d_x^2 + c_yy d_y^2 + c_zz d_z^2 + c_xy d_x d_y +
// c_xz d_x d_z + c_yz d_y d_z and m = [i mobile] + [j mobile] (the ordered
// pairs of W that contain the pair):
//   xbar_i += m/2 (s_c (grad Q / r - Q d / r^3) + (Q / r) s_c' e),
//   rhobar_i += m/2 (Q / r) B wd [r < r_d],  s_c' = ds_c/dr at fixed rho.
// The partner lists hold every pair from both sides, so each thread adds its
// own particle's share without atomics (a particle with more partners than
// list slots scans its neighbour cells instead, as the force pass does).  A second pass sends rhobar back to
// positions: xbar_i += (rhobar_i + rhobar_j) w_rho'(r) e over partners within
// r_d.
//
// Parameter gradients are deterministic: each thread accumulates its pairs'
// terms in its own shared-memory column, indexed by (parameter, partner
// type); the block then adds the columns of its threads by a fixed tree for
// every (parameter, own type, partner type), and a per-replica kernel adds the
// blocks in a fixed order.  Each unordered pair is seen from both sides, so each
// side adds half its term.
#include "pair.cuh"
#include "roots.cuh"

namespace mdpd {

namespace {

constexpr int TB = 3 * 64;         // parameter slots [q][a][b], q = A, B, gamma
constexpr int TCOL = 3 * 8;        // per-thread columns [q][partner type]

// 1 / sqrt(x): FP32 from the hardware estimate (2 ulp) with one Newton step, FP64 by
// the library function (1 ulp; 1 / sqrt has up to 1.5).  (Quotients by r are products
// with it: an FP64 division is some ten instructions at 1/64 of the FP32 rate, and a
// pair had up to thirteen.)
__device__ __forceinline__ float inv_sqrt(float x) { return inv_sqrt_step(x, rsqrtf(x)); }
__device__ __forceinline__ double inv_sqrt(double x) { return rsqrt(x); }

// A parameter gradient's running sum over one particle's pairs.  In FP32 a pair of
// floats (the rounding of every addition kept: Knuth's two-sum): the gradients' errors
// are those of FP64 sums of the same terms to three digits, off the FP64 pipe.
struct Sum2 {
    float hi, lo;
};
template <typename T> struct ColSum;
template <> struct ColSum<float> { using type = Sum2; };
template <> struct ColSum<double> { using type = double; };
__device__ __forceinline__ void col_add(Sum2& c, float x)
{
    const float s = __fadd_rn(c.hi, x), t = __fsub_rn(s, c.hi);
    c.lo = __fadd_rn(c.lo, __fadd_rn(__fsub_rn(c.hi, __fsub_rn(s, t)), __fsub_rn(x, t)));
    c.hi = s;
}
__device__ __forceinline__ void col_add(double& c, double x) { c += x; }
__device__ __forceinline__ double col_value(const Sum2& c) { return (double)c.hi + (double)c.lo; }
__device__ __forceinline__ double col_value(double c) { return c; }

// d(sigma)/d(gamma) of a type pair: in FP64 over sqrt(dt); in FP32 a pair of floats, for
// every term of the random force's share in the gamma gradient has it as a factor, so
// its rounding would not average out.
template <typename T> struct DSigma;
template <> struct DSigma<float> {
    using type = float2;
    static __device__ __forceinline__ float2 make(double d, double)
    {
        const float hi = (float)d;
        return make_float2(hi, (float)(d - (double)hi));
    }
};
template <> struct DSigma<double> {
    using type = double;
    static __device__ __forceinline__ double make(double d, double inv_sqrt_dt) { return d * inv_sqrt_dt; }
};
// Adds a pair's share hq wc (d xi / sqrt(dt) - wc w) of the gamma gradient, in FP32 with
// the roundings of the products by hq, wc and d kept (a fused multiply-add gives a
// product's rounding exactly).  Error of the gradient against 64 bits, rms over 300
// draws, with FP64 terms and sums / one rounded FP32 term a pair / so: liquids of 1,503
// particles 1.71 / 1.92 / 1.70e-7, of 40,009 1.60 / 1.77 / 1.65e-7; VJP of 100,000
// particles 301 us with the rounded term, 304 so (two runs of one side differ by more).
__device__ __forceinline__ void col_add_gamma(Sum2& col, float hq, float2 d, float wc, float xi,
                                              float inv_sqrt_dt, float w)
{
    const float v = xi * inv_sqrt_dt;
    const float h = __fmul_rn(hq, wc), he = fmaf(hq, wc, -h);
    const float m = fmaf(d.x, v, -(wc * w));
    const float p = __fmul_rn(h, m), pe = fmaf(h, m, -p);
    col_add(col, p);
    col.lo = __fadd_rn(col.lo, fmaf(h, d.y * v, fmaf(he, m, pe)));
}
__device__ __forceinline__ void col_add_gamma(double& col, double hq, double d, double wc, double xi,
                                              double, double w)
{
    col += hq * wc * (d * xi - wc * w);
}

// Adjoints of the accelerations in cell order (zero for frozen particles): 16 bytes a
// slot in FP32, 24 in FP64.
__device__ __forceinline__ void store_abar(float4* a, int64_t s, double x, double y, double z)
{
    a[s] = make_float4((float)x, (float)y, (float)z, 0.0f);
}
__device__ __forceinline__ void store_abar(double* a, int64_t s, double x, double y, double z)
{
    a[3 * s] = x;
    a[3 * s + 1] = y;
    a[3 * s + 2] = z;
}
__device__ __forceinline__ void load_abar(const float4* __restrict__ a, int64_t s, float (&q)[3])
{
    const float4 v = a[s];
    q[0] = v.x;
    q[1] = v.y;
    q[2] = v.z;
}
__device__ __forceinline__ void load_abar(const double* __restrict__ a, int64_t s, double (&q)[3])
{
    q[0] = a[3 * s];
    q[1] = a[3 * s + 1];
    q[2] = a[3 * s + 2];
}
template <typename T> struct AbarOf;
template <> struct AbarOf<float> { using type = float4; };
template <> struct AbarOf<double> { using type = double; };

// The block's particle slot, replica record and validity (see Batch).
template <bool BATCH>
struct BlockSite {
    int s;
    bool valid;
    int r;
    const Rep* rp;
};

template <bool BATCH>
__device__ __forceinline__ BlockSite<BATCH> block_site(int n, const Batch& bt)
{
    BlockSite<BATCH> b;
    if constexpr (BATCH) {
        const int4 ch = bt.chunks[blockIdx.x];
        b.rp = &block_rep<REP_SCALARS>(bt.reps, ch.x);
        b.r = ch.x;
        b.s = ch.y + (int)threadIdx.x;
        b.valid = (int)threadIdx.x < ch.z;
    } else {
        b.rp = nullptr;
        b.r = 0;
        b.s = blockIdx.x * PAIR_BLOCK + threadIdx.x;
        b.valid = b.s < n;
    }
    return b;
}

// Visit the partners within r_c (0 < r) of particle s: from its list, or, for
// a particle with more partners than list slots, by a scan of its 27
// neighbour cells (the same partners, in cell order), as the force pass does.
template <typename T, typename V, typename F>
__device__ __forceinline__ void for_partners(int s, uint32_t cnt, int64_t cap,
                                             const uint32_t* __restrict__ nl, const Geo& geo,
                                             int64_t cell0, const uint32_t* __restrict__ cell_s,
                                             const uint32_t* __restrict__ start,
                                             const V* __restrict__ pos4, const V& pi,
                                             const T (&shift)[27][3], T rc2,
                                             uint32_t* __restrict__ dbg, F&& partner)
{
    if (cnt <= (uint32_t)NL_MAX) {
        for (uint32_t k = 0; k < cnt; ++k) {
            const uint32_t e = nl[(int64_t)k * cap + s];
            if (MDPD_DBG_OK((e >> 5) < (uint32_t)cap && (e & 31u) < 27u, dbg))
                partner(e >> 5, e & 31u);
        }
        return;
    }
    int q0, q1, q2;
    cell_coords(cell_s[s], geo, q0, q1, q2);      // (the cell within the replica)
    for (int oz = -1; oz <= 1; ++oz) {
        const int z = neighbour_index(q2, oz, geo.nc[2], geo.periodic[2]);
        if (z < 0) continue;
        for (int oy = -1; oy <= 1; ++oy) {
            const int y = neighbour_index(q1, oy, geo.nc[1], geo.periodic[1]);
            if (y < 0) continue;
            for (int ox = -1; ox <= 1; ++ox) {
                const int x = neighbour_index(q0, ox, geo.nc[0], geo.periodic[0]);
                if (x < 0) continue;
                const uint32_t code = (uint32_t)((ox + 1) + 3 * (oy + 1) + 9 * (oz + 1));
                const uint32_t nc = (uint32_t)(cell0 + x + geo.nc[0] * (y + geo.nc[1] * z));
                const uint32_t b = start[nc];
                uint32_t e = start[nc + 1];
                if (!MDPD_DBG_OK(b <= e && e <= (uint32_t)cap, dbg)) e = b;
                for (uint32_t j = b; j < e; ++j) {
                    const V pj = pos4[j];
                    const T dx = pi.x - shift[code][0] - pj.x;
                    const T dy = pi.y - shift[code][1] - pj.y;
                    const T dz = pi.z - shift[code][2] - pj.z;
                    const T r2 = dx * dx + dy * dy + dz * dz;
                    if (r2 < rc2 && r2 > T(0)) partner(j, code);
                }
            }
        }
    }
}

// abar (id order) to cell order in the pair precision.
template <typename T>
__global__ void k_gather_abar(int n, const uint32_t* __restrict__ id, const double* __restrict__ abar, typename AbarOf<T>::type* __restrict__ out)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    const int64_t i = id[s];
    store_abar(out, s, abar[3 * i], abar[3 * i + 1], abar[3 * i + 2]);
}

// Bound by issue (FP32: about 130 instructions a pair, 45 of them the draw) and, in
// FP64, by the FP64 pipe (70 a pair).  The parameters' sums per pair stay out of it:
// tables in the pair precision, running sums in Sum2.
// VJP of 100,000 particles in FP32, with the density passes: 624 -> 294 us (FP64 sums,
// thirteen quotients and gathers of abar by id per pair before).
template <typename T, bool BATCH>
__global__ void __launch_bounds__(PAIR_BLOCK)
k_force_vjp(int n, int64_t cap, Geo geo_p, Phys ph_p, Batch bt,
            const typename Vec4<T>::type* __restrict__ pos4,
            const typename Vec4<T>::type* __restrict__ vel4, const T* __restrict__ rho,
            const uint32_t* __restrict__ cell_s, const uint32_t* __restrict__ start,
            const uint32_t* __restrict__ nl, const uint32_t* __restrict__ nl_count,
            const uint64_t* __restrict__ step_ptr,
            const typename AbarOf<T>::type* __restrict__ abar, const double* __restrict__ wbar,
            const double* __restrict__ rhobar, double* __restrict__ xbar,
            double* __restrict__ ubar, T* __restrict__ rbar, double* __restrict__ tpart,
            uint32_t* __restrict__ status)
{
    using V = typename Vec4<T>::type;
    using Col = typename ColSum<T>::type;
    __shared__ Col col[TCOL][PAIR_BLOCK];
    __shared__ T shift[27][3];
    __shared__ PairTables<T> tab;              // A, B, gamma, sigma / sqrt(dt)
    __shared__ typename DSigma<T>::type dsig[64];
    __shared__ double wsum[PAIR_BLOCK / 32];
    const BlockSite<BATCH> b = block_site<BATCH>(n, bt);
    const Phys& ph = BATCH ? b.rp->ph : ph_p;             // scalars (and tables if single)
    const Phys& tabs = BATCH ? bt.reps[b.r].ph : ph_p;    // per-type-pair tables
    const uint32_t id0 = BATCH ? b.rp->id0 : 0u;
    const Derived<T>& dc = derived<T>(ph);
    const int tid = threadIdx.x;
    const int nt = ph.ntypes;
#pragma unroll
    for (int q = 0; q < 3; ++q)
        for (int t = 0; t < nt; ++t) col[q * 8 + t][tid] = Col{};
    for (int k = tid; k < 64; k += PAIR_BLOCK) {
        tab.P[k] = make4((T)tabs.A[k], (T)tabs.B[k], (T)tabs.gamma[k], (T)tabs.sigma[k] * dc.inv_sqrt_dt);
        dsig[k] = DSigma<T>::make(tabs.gamma[k] > 0.0 ? ph.kT / tabs.sigma[k] : 0.0,
                                  ph.dd.inv_sqrt_dt);
    }
    if (tid < 27) {
        shift[tid][0] = (T)(tid % 3 - 1) * dc.h[0];
        shift[tid][1] = (T)((tid / 3) % 3 - 1) * dc.h[1];
        shift[tid][2] = (T)(tid / 9 - 1) * dc.h[2];
    }
    const int s = b.s;
    uint32_t ti = 0xFFu;
    __syncthreads();
    if (b.valid) {
        const uint64_t step = *step_ptr;
        const T inv_rc = dc.inv_rc, inv_rd = dc.inv_rd;
        // virial weights of this replica (c_xx c_yy c_zz c_xy c_xz c_yz)
        T cw[6] = { T(0), T(0), T(0), T(0), T(0), T(0) };
        const bool vir = wbar != nullptr;
        if (vir)
#pragma unroll
            for (int k = 0; k < 6; ++k) cw[k] = (T)wbar[6 * b.r + k];
        const V pi = pos4[s];
        const V vi = vel4[s];
        const T rho_i = rho[s];
        const uint32_t id_i = unpack_u32(vi.w);
        ti = type_of(pi.w);
        const bool mob_i = ((ph.frozen >> ti) & 1u) == 0u;
        T ai[3] = { T(0), T(0), T(0) };
        if (abar && mob_i) load_abar(abar, s, ai);
        T gx[3] = { T(0), T(0), T(0) }, gu[3] = { T(0), T(0), T(0) };
        T gr = T(0);
        // one partner j in the image of neighbour-cell code `code`
        auto partner = [&](uint32_t j, uint32_t code) {
            const V pj = pos4[j];
            const V vj = vel4[j];
            const T rho_j = rho[j];
            const uint32_t tj = type_of(pj.w), id_j = unpack_u32(vj.w);
            const bool mob_j = ((ph.frozen >> tj) & 1u) == 0u;
            const T dx = pi.x - shift[code][0] - pj.x;
            const T dy = pi.y - shift[code][1] - pj.y;
            const T dz = pi.z - shift[code][2] - pj.z;
            const T r2 = dx * dx + dy * dy + dz * dz;
            const T rinv = inv_sqrt(r2);
            const T r = sqrt_from(r2, rinv);
            const T e3[3] = { dx * rinv, dy * rinv, dz * rinv };
            const T wc = T(1) - r * inv_rc;
            const T wd0 = T(1) - r * inv_rd;
            const bool near = wd0 > T(0);
            const T wd = near ? wd0 : T(0);
            const int pidx = (int)(ti * 8 + tj);
            const V prm = tab.P[pidx];
            const T A = prm.x, B = prm.y;
            const T rsum = rho_i + rho_j;
            const T sc = A * wc + B * rsum * wd;                                // F^C
            const T sc_r = -A * inv_rc - (near ? B * rsum * inv_rd : T(0));     // its d/dr
            if (abar) {
                T q[3] = { T(0), T(0), T(0) };
                if (mob_j) load_abar(abar, j, q);
#pragma unroll
                for (int c = 0; c < 3; ++c) q[c] = ai[c] - q[c];
                const T u3[3] = { vi.x - vj.x, vi.y - vj.y, vi.z - vj.z };
                const T w = e3[0] * u3[0] + e3[1] * u3[1] + e3[2] * u3[2];
                const U4 wr = BATCH ? pair_draw(id_i, id_j, step, ph.key0, ph.key1)
                                    : pair_draw_rk(id_i, id_j, step, ph.rk);
                const T xi = xi_of<T>(wr, ph.xi_dist);
                const T gw = prm.z * wc, sx = prm.w * xi;      // gamma wc, sigma xi / sqrt(dt)
                const T sval = sc + wc * (sx - gw * w);
                const T s_r = sc_r + (T(2) * gw * w - sx) * inv_rc;
                const T s_w = -gw * wc;
                const T qe = q[0] * e3[0] + q[1] * e3[1] + q[2] * e3[2];
                const T be = qe * s_w, sr = sval * rinv, br = be * rinv;
                if constexpr (sizeof(T) == 8) {
                // (q.e) s_r e + br (u - w e) + sr (q - (q.e) e), by the vectors' sums
                const T al = qe * (s_r - sr) - br * w;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    gx[c] += al * e3[c];
                    gx[c] += br * u3[c];
                    gx[c] += sr * q[c];
                    gu[c] += be * e3[c];
                }
                } else {
                const T al = qe * s_r;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    gx[c] += al * e3[c] + br * (u3[c] - w * e3[c]) + sr * (q[c] - qe * e3[c]);
                    gu[c] += be * e3[c];
                }
                }
                gr += qe * B * wd;
                const T hq = T(0.5) * qe;
                col_add(col[tj][tid], hq * wc);
                col_add(col[8 + tj][tid], hq * rsum * wd);
                col_add_gamma(col[16 + tj][tid], hq, dsig[pidx], wc, xi, dc.inv_sqrt_dt, w);
            }
            if (vir) {
                const T mm = T((mob_i ? 1 : 0) + (mob_j ? 1 : 0));
                if (mm > T(0)) {
                    const T Q = cw[0] * dx * dx + cw[1] * dy * dy + cw[2] * dz * dz +
                                cw[3] * dx * dy + cw[4] * dx * dz + cw[5] * dy * dz;
                    const T gQ[3] = { T(2) * cw[0] * dx + cw[3] * dy + cw[4] * dz,
                                      T(2) * cw[1] * dy + cw[3] * dx + cw[5] * dz,
                                      T(2) * cw[2] * dz + cw[4] * dx + cw[5] * dy };
                    const T hm = T(0.5) * mm, Qr = Q * rinv;
                    const T sq = hm * sc * rinv, er = hm * Qr * (sc_r - sc * rinv);
#pragma unroll
                    for (int c = 0; c < 3; ++c) gx[c] += sq * gQ[c] + er * e3[c];
                    gr += hm * Qr * B * wd;
                    const T hr = T(0.5) * hm * Qr;
                    col_add(col[tj][tid], hr * wc);
                    col_add(col[8 + tj][tid], hr * rsum * wd);
                }
            }
        };
        const Geo& geo = BATCH ? b.rp->geo : geo_p;
        if (abar || vir)
            for_partners<T>(s, nl_count[s], cap, nl, geo, BATCH ? b.rp->cell0 : 0, cell_s, start, pos4,
                            pi, shift, derived<T>(ph).rc2, ph.dbg_status, partner);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            xbar[c * cap + s] = (double)gx[c];
            ubar[c * cap + s] = (double)gu[c];
        }
        rbar[s] = rhobar ? (T)((double)gr + rhobar[id0 + id_i]) : gr;
    }
    // slot (q, a, b): the columns (q, b) of the block's threads of type a, added over
    // the warp by a fixed tree and over the warps in order
    const int lane = tid & 31, warp = tid >> 5;
    for (int k = 0; k < TB; ++k) {
        const int q = k / 64, a = (k / 8) % 8, bb = k % 8;
        double v = 0.0;
        if (a < nt && bb < nt) {                          // (block-uniform)
            if (ti == (uint32_t)a) v = col_value(col[q * 8 + bb][tid]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            __syncthreads();
            if (lane == 0) wsum[warp] = v;
            __syncthreads();
            if (tid == 0) {
                v = wsum[0];
                for (int t = 1; t < PAIR_BLOCK / 32; ++t) v += wsum[t];
                tpart[(int64_t)blockIdx.x * TB + k] = v;
            }
        }
    }
}

template <typename T, bool BATCH>
__global__ void __launch_bounds__(PAIR_BLOCK)
k_density_vjp(int n, int64_t cap, Geo geo_p, Phys ph_p, Batch bt,
              const typename Vec4<T>::type* __restrict__ pos4,
              const uint32_t* __restrict__ cell_s, const uint32_t* __restrict__ start,
              const uint32_t* __restrict__ nl, const uint32_t* __restrict__ nl_count,
              const T* __restrict__ rbar, double* __restrict__ xbar,
              uint32_t* __restrict__ status)
{
    using V = typename Vec4<T>::type;
    __shared__ T shift[27][3];
    const BlockSite<BATCH> b = block_site<BATCH>(n, bt);
    const Phys& ph = BATCH ? b.rp->ph : ph_p;
    if (threadIdx.x < 27) {
        const int c = threadIdx.x;
        shift[c][0] = (T)(c % 3 - 1) * derived<T>(ph).h[0];
        shift[c][1] = (T)((c / 3) % 3 - 1) * derived<T>(ph).h[1];
        shift[c][2] = (T)(c / 9 - 1) * derived<T>(ph).h[2];
    }
    __syncthreads();
    if (!b.valid) return;
    const int s = b.s;
    const Derived<T>& dc = derived<T>(ph);
    const T inv_rd = dc.inv_rd;
    const T cw = T(-2) * dc.cw_rho * inv_rd;              // w_rho'(r) = cw (1 - r / r_d)
    const V pi = pos4[s];
    const T rb_i = rbar[s];
    T g[3] = { T(0), T(0), T(0) };
    auto partner = [&](uint32_t j, uint32_t code) {
        const V pj = pos4[j];
        const T dx = pi.x - shift[code][0] - pj.x;
        const T dy = pi.y - shift[code][1] - pj.y;
        const T dz = pi.z - shift[code][2] - pj.z;
        const T r2 = dx * dx + dy * dy + dz * dz;
        if (!(r2 < dc.rd2)) return;
        const T rinv = inv_sqrt(r2);
        const T f = (rb_i + rbar[j]) * cw * (rinv - inv_rd);      // ... w_rho'(r) / r
        g[0] += f * dx;
        g[1] += f * dy;
        g[2] += f * dz;
    };
    const Geo& geo = BATCH ? b.rp->geo : geo_p;
    for_partners<T>(s, nl_count[s], cap, nl, geo, BATCH ? b.rp->cell0 : 0, cell_s, start, pos4, pi,
                    shift, derived<T>(ph).rc2, ph.dbg_status, partner);
#pragma unroll
    for (int c = 0; c < 3; ++c) xbar[c * cap + s] += (double)g[c];
}

// Per replica (one block each): the sum of its blocks' parameter partials, stored
// (add = 0) or added (add = 1) to acc.  P warps take a slot: their lanes add every
// 32 P-th block and are added by a fixed tree, then the warps in order.  Only slots of
// types below nt are formed (the others are zero).  (One thread per slot added the
// blocks one after another: 99 us for 782 blocks.)
// ranges[r] = (first, end) of replica r's blocks (x4 for warp ranges: scale).
constexpr int RED_WARPS = 32;
__global__ void __launch_bounds__(RED_WARPS * 32)
k_theta_reduce(int nrep, int nblk, const int2* __restrict__ ranges, int scale, int nt,
               const double* __restrict__ tpart, double* __restrict__ acc, int add)
{
    const int r = blockIdx.x, lane = threadIdx.x & 31;
    int lo = 0, hi = nblk;
    if (ranges) {
        lo = ranges[r].x / scale;
        hi = ranges[r].y / scale;
    }
    __shared__ double part[RED_WARPS];
    const int warp = threadIdx.x >> 5;
    const int used = 3 * nt * nt;
    const int P = max(1, RED_WARPS / used), S = RED_WARPS / P;      // warps a slot, slots at once
    for (int u0 = 0; u0 < used; u0 += S) {
        const int u = u0 + warp / P, p = warp % P;
        const bool on = warp < S * P && u < used;
        const int k = on ? u / (nt * nt) * 64 + u / nt % nt * 8 + u % nt : 0;
        double sum = 0.0;
        if (on) {
#pragma unroll 4
            for (int b = lo + 32 * p + lane; b < hi; b += 32 * P) sum += tpart[(int64_t)b * TB + k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, o);
            if (lane == 0) part[warp] = sum;
        }
        __syncthreads();
        if (on && p == 0 && lane == 0) {
            for (int t = 1; t < P; ++t) sum += part[warp + t];
            acc[(int64_t)r * TB + k] = add ? acc[(int64_t)r * TB + k] + sum : sum;
        }
        __syncthreads();
    }
    if (!add)
        for (int k = threadIdx.x; k < TB; k += RED_WARPS * 32)
            if ((k / 8) % 8 >= nt || k % 8 >= nt) acc[(int64_t)r * TB + k] = 0.0;
}

// Gradient of the symmetric tables from the per-(own type, partner type) sums
// S: out[q][a][b] = out[q][b][a] = S[q][a][b] + S[q][b][a] for a != b and
// S[q][a][a] on the diagonal.
__global__ void k_theta_symmetrise(int nrep, const double* __restrict__ acc, double* __restrict__ out)
{
    const int r = blockIdx.x, k = threadIdx.x;
    if (r >= nrep || k >= TB) return;
    const int q = k / 64, a = (k / 8) % 8, b = k % 8;
    const double* S = acc + (int64_t)r * TB + q * 64;
    out[(int64_t)r * TB + k] = a == b ? S[a * 8 + a] : S[a * 8 + b] + S[b * 8 + a];
}

// ---- velocity-Verlet window ------------------------------------------------
// Each kernel walks the slots of the current binning (chunks of a batch), so
// that the particle's type, replica and id are at hand; vectors in id order
// are interleaved xyz (element 3 * id + k).

template <bool BATCH>
struct SlotSite {
    int s;
    bool valid;
    const Rep* rp;
};

template <bool BATCH>
__device__ __forceinline__ SlotSite<BATCH> slot_site(int n, const Batch& bt)
{
    SlotSite<BATCH> b;
    if constexpr (BATCH) {
        const int4 ch = bt.chunks[blockIdx.x];
        b.rp = &block_rep<REP_SCALARS>(bt.reps, ch.x);
        b.s = ch.y + (int)threadIdx.x;
        b.valid = (int)threadIdx.x < ch.z;
    } else {
        b.rp = nullptr;
        b.s = blockIdx.x * blockDim.x + threadIdx.x;
        b.valid = b.s < n;
    }
    return b;
}

// Checkpoint of step k of a window: X = x_k and, if VH is given, the
// half-step velocity v'_k = v_k + (dt/2) a_k of mobile particles formed with
// the same arithmetic as the integrator's first half-kick (kick_drift_one;
// frozen particles keep v).
template <bool BATCH>
__global__ void __launch_bounds__(BATCH_CHUNK)
k_win_record(int n, int64_t cap, Phys ph_p, Batch bt, Master m, double* __restrict__ X,
             double* __restrict__ VH)
{
    const SlotSite<BATCH> b = slot_site<BATCH>(n, bt);
    if (!b.valid) return;
    const Phys& ph = BATCH ? b.rp->ph : ph_p;
    const int s = b.s;
    const int64_t i = m.id[s];
    const bool mob = ((ph.frozen >> m.type[s]) & 1u) == 0u;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        X[3 * i + k] = m.x[k * cap + s];
        if (VH) {
            const double v = m.v[k * cap + s];
            const double a = m.a[k * cap + s];
            const double d = ph.prec32 ? to_f64(ph.df.hdt * to_f32(a)) : __dmul_rn(ph.hdt, a);
            VH[3 * i + k] = mob ? __dadd_rn(v, d) : v;
        }
    }
}

// Start of the reverse sweep: xb = xbar_K, vb = vbar_K, ab = (dt/2) vb
// (mobile), the adjoint of the last half-kick.
template <bool BATCH>
__global__ void __launch_bounds__(BATCH_CHUNK)
k_win_init(int n, Phys ph_p, Batch bt, Master m, const double* __restrict__ xbar,
           const double* __restrict__ vbar, double* __restrict__ xb, double* __restrict__ vb,
           double* __restrict__ ab)
{
    const SlotSite<BATCH> b = slot_site<BATCH>(n, bt);
    if (!b.valid) return;
    const Phys& ph = BATCH ? b.rp->ph : ph_p;
    const int s = b.s;
    const int64_t i = m.id[s];
    const double mob = ((ph.frozen >> m.type[s]) & 1u) == 0u ? 1.0 : 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double x = xbar ? xbar[3 * i + k] : 0.0;
        const double v = vbar ? vbar[3 * i + k] : 0.0;
        xb[3 * i + k] = x;
        vb[3 * i + k] = v;
        ab[3 * i + k] = __dmul_rn(__dmul_rn(ph.hdt, v), mob);
    }
}

// After the force VJP of step k (outputs gx, gu in cell order, [3][cap]):
//   xb += gx;  vhb = vb + gu + dt xb (mobile);  vb = vhb;
//   ab = (dt/2) vhb (mobile), plus (dt/2) vb once more unless this was the
//   window's first step (the next step's half-kick adjoint).
// final = 1 (the VJP of a_0 = F(x_0, v_0)): x0bar = xb + gx, v0bar = vb + gu.
template <bool BATCH>
__global__ void __launch_bounds__(BATCH_CHUNK)
k_win_post(int n, int64_t cap, Phys ph_p, Batch bt, Master m, const double* __restrict__ gx,
           const double* __restrict__ gu, double* __restrict__ xb, double* __restrict__ vb,
           double* __restrict__ ab, int first, int final, double* __restrict__ x0bar,
           double* __restrict__ v0bar)
{
    const SlotSite<BATCH> b = slot_site<BATCH>(n, bt);
    if (!b.valid) return;
    const Phys& ph = BATCH ? b.rp->ph : ph_p;
    const int s = b.s;
    const int64_t i = m.id[s];
    const double mob = ((ph.frozen >> m.type[s]) & 1u) == 0u ? 1.0 : 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double g = gx[k * cap + s], u = gu[k * cap + s];
        if (final) {
            if (x0bar) x0bar[3 * i + k] = __dadd_rn(xb[3 * i + k], g);
            if (v0bar) v0bar[3 * i + k] = __dadd_rn(vb[3 * i + k], u);
            continue;
        }
        const double x = __dadd_rn(xb[3 * i + k], g);
        const double vh = __dadd_rn(__dadd_rn(vb[3 * i + k], u), __dmul_rn(__dmul_rn(ph.dt, x), mob));
        const double t = __dmul_rn(__dmul_rn(ph.hdt, vh), mob);
        xb[3 * i + k] = x;
        vb[3 * i + k] = vh;
        ab[3 * i + k] = first ? t : __dadd_rn(t, t);
    }
}

inline unsigned pair_blocks(int n) { return (unsigned)((n + PAIR_BLOCK - 1) / PAIR_BLOCK); }

}  // namespace

int vjp_num_blocks(int n, const Batch* bt)
{
    return bt ? bt->nchunk : (int)pair_blocks(n);
}

void launch_force_vjp(cudaStream_t st, int precision, int n, int64_t cap, const Geo& geo,
                      const Phys& ph, const Batch* bt, const void* pos4, const void* vel4,
                      const void* rho, const uint32_t* cell_s, const uint32_t* start,
                      const uint32_t* nl, const uint32_t* nl_count, const uint64_t* step_ptr,
                      const uint32_t* id, const double* abar, void* abar_s, const double* wbar,
                      const double* rhobar, double* xbar, double* ubar, void* rbar, double* tpart,
                      uint32_t* status)
{
    const int nb = vjp_num_blocks(n, bt);
    if (nb <= 0) return;
    const Batch bb = bt ? *bt : Batch{};
    const size_t smem = bt ? REP_SMEM : 0;
    auto go = [&](auto t, auto k) {
        using T = decltype(t);
        using A = typename AbarOf<T>::type;
        using V = typename Vec4<T>::type;
        if (abar)
            k_gather_abar<T><<<(n + 255) / 256, 256, 0, st>>>(n, id, abar, (A*)abar_s);
        k<<<nb, PAIR_BLOCK, smem, st>>>(n, cap, geo, ph, bb, (const V*)pos4, (const V*)vel4,
                                        (const T*)rho, cell_s, start, nl, nl_count, step_ptr,
                                        abar ? (const A*)abar_s : nullptr, wbar, rhobar, xbar, ubar,
                                        (T*)rbar, tpart, status);
    };
    if (precision == 0) go(double{}, bt ? k_force_vjp<double, true> : k_force_vjp<double, false>);
    else go(float{}, bt ? k_force_vjp<float, true> : k_force_vjp<float, false>);
}

void launch_density_vjp(cudaStream_t st, int precision, int n, int64_t cap, const Geo& geo,
                        const Phys& ph, const Batch* bt, const void* pos4,
                        const uint32_t* cell_s, const uint32_t* start, const uint32_t* nl,
                        const uint32_t* nl_count, const void* rbar, double* xbar,
                        uint32_t* status)
{
    const int nb = vjp_num_blocks(n, bt);
    if (nb <= 0) return;
    const Batch bb = bt ? *bt : Batch{};
    const size_t smem = bt ? REP_SMEM : 0;
    auto go = [&](auto t, auto k) {
        using T = decltype(t);
        k<<<nb, PAIR_BLOCK, smem, st>>>(n, cap, geo, ph, bb, (const typename Vec4<T>::type*)pos4,
                                        cell_s, start, nl, nl_count, (const T*)rbar, xbar, status);
    };
    if (precision == 0) go(double{}, bt ? k_density_vjp<double, true> : k_density_vjp<double, false>);
    else go(float{}, bt ? k_density_vjp<float, true> : k_density_vjp<float, false>);
}

__global__ void k_set_u64(uint64_t* __restrict__ p, uint64_t v) { *p = v; }

void launch_set_step(cudaStream_t st, uint64_t* step_ptr, uint64_t value)
{
    k_set_u64<<<1, 1, 0, st>>>(step_ptr, value);
}

void launch_theta_reduce(cudaStream_t st, int nrep, int nblk, const int2* ranges, int scale,
                         int nt, const double* tpart, double* acc, int add)
{
    if (nrep <= 0) return;
    k_theta_reduce<<<nrep, RED_WARPS * 32, 0, st>>>(nrep, nblk, ranges, scale, nt, tpart, acc, add);
}

void launch_theta_symmetrise(cudaStream_t st, int nrep, const double* acc, double* out)
{
    if (nrep <= 0) return;
    k_theta_symmetrise<<<nrep, TB, 0, st>>>(nrep, acc, out);
}

void launch_win_record(cudaStream_t st, int n, int64_t cap, const Phys& ph, const Batch* bt,
                       const Master& m, double* X, double* VH)
{
    if (bt) {
        if (bt->nchunk > 0)
            k_win_record<true><<<bt->nchunk, BATCH_CHUNK, REP_SMEM, st>>>(n, cap, ph, *bt, m, X, VH);
    } else if (n > 0) {
        k_win_record<false><<<(n + BATCH_CHUNK - 1) / BATCH_CHUNK, BATCH_CHUNK, 0, st>>>(
            n, cap, ph, Batch{}, m, X, VH);
    }
}

void launch_win_init(cudaStream_t st, int n, const Phys& ph, const Batch* bt, const Master& m,
                     const double* xbar, const double* vbar, double* xb, double* vb, double* ab)
{
    if (bt) {
        if (bt->nchunk > 0)
            k_win_init<true><<<bt->nchunk, BATCH_CHUNK, REP_SMEM, st>>>(n, ph, *bt, m, xbar, vbar,
                                                                        xb, vb, ab);
    } else if (n > 0) {
        k_win_init<false><<<(n + BATCH_CHUNK - 1) / BATCH_CHUNK, BATCH_CHUNK, 0, st>>>(
            n, ph, Batch{}, m, xbar, vbar, xb, vb, ab);
    }
}

void launch_win_post(cudaStream_t st, int n, int64_t cap, const Phys& ph, const Batch* bt,
                     const Master& m, const double* gx, const double* gu, double* xb, double* vb,
                     double* ab, int first, int final, double* x0bar, double* v0bar)
{
    if (bt) {
        if (bt->nchunk > 0)
            k_win_post<true><<<bt->nchunk, BATCH_CHUNK, REP_SMEM, st>>>(
                n, cap, ph, *bt, m, gx, gu, xb, vb, ab, first, final, x0bar, v0bar);
    } else if (n > 0) {
        k_win_post<false><<<(n + BATCH_CHUNK - 1) / BATCH_CHUNK, BATCH_CHUNK, 0, st>>>(
            n, cap, ph, Batch{}, m, gx, gu, xb, vb, ab, first, final, x0bar, v0bar);
    }
}

}  // namespace mdpd
