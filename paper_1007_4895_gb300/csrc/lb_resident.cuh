/*
 * lb_resident.cuh -- several time steps of small lattices in one launch, with the state
 * in shared memory from the first step to the last.
 *
 * What bounds small lattices is latency: a step of a few thousand nodes takes a launch, a
 * trip to L2 or DRAM per population and a chain of 9 to 36 populations in every thread,
 * on a few warps. Here a block (or a cluster of blocks, each with a band of rows) loads a
 * lattice, or a bundle of small lattices, once, and does per step
 *   1. every node's moments in population order (Eq. (demoeq)), after the diffuse-wall
 *      fill of wall rows (Sec. 3.2), and the node's collision coefficients;
 *   2. the mode-B views of rows next to the other set (Sec. 2.2);
 *   3. the Sec. 3.1 update, in units of 32 quads (nodes) x a group of populations, so that
 *      the populations of one node run on several warps at once;
 * with block barriers between (cluster barriers where rows of another block are read).
 * The level is stored as planes [population][row slot][x]; the new planes go to spare
 * planes, the old ones become spare: with K spare planes a step takes ceil(Q / K) rounds
 * with a barrier each (K = Q: two full levels, one round). A row's neighbours are row
 * slots from a table, so walls (ghost node = wall node), periodic images, rows of the
 * other set (views) and rows of the next block (pushed there by their owner through
 * distributed shared memory when they are updated) cost no index logic and no copies.
 *
 * PAIR: quads in the paired arithmetic of layout 9 (lb_pair.cuh), the same bits as layout
 * 9; else one node per lane in layout 0's arithmetic, the same bits as layout 0.
 */
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <atomic>
#include <type_traits>

#include "lb_pair.cuh"
#include "lb_resident_host.h"

namespace lbk {

/* One block's view of its lattices, in shared memory */
template <typename R>
struct ResLat {
    R rho0, dt, kn_rho, tau_shift, gx, gy;
    R uw_x[2], uw_y[2], kdiff[2][2], kout[2][2];
    int tau_const, pad;
};

/* Constants of one population: the paired arithmetic's are RingPop */
template <typename R>
struct alignas(16) ResPop {
    R cx, cy, crx, cry, kx, ky, w, winv, wcx, wcy, wxx, wxy, wyy, hxx, hxy, hyy;
};

template <bool PAIR, typename R>
struct ResPopOf {
    using type = RingPop;
    static __device__ __forceinline__ R w(const RingPop &p) { return p.w2.x; }
    static __device__ __forceinline__ R winv(const RingPop &p) { return p.winv2.x; }
    static __device__ __forceinline__ R cx(const RingPop &p) { return p.cx2.x; }
    static __device__ __forceinline__ R cy(const RingPop &p) { return p.cy2.x; }
    static __device__ __forceinline__ R wcx(const RingPop &p) { return p.wcx2.x; }
    static __device__ __forceinline__ R wcy(const RingPop &p) { return p.wcy2.x; }
};
template <typename R>
struct ResPopOf<false, R> {
    using type = ResPop<R>;
    static __device__ __forceinline__ R w(const ResPop<R> &p) { return p.w; }
    static __device__ __forceinline__ R winv(const ResPop<R> &p) { return p.winv; }
    static __device__ __forceinline__ R cx(const ResPop<R> &p) { return p.cx; }
    static __device__ __forceinline__ R cy(const ResPop<R> &p) { return p.cy; }
    static __device__ __forceinline__ R wcx(const ResPop<R> &p) { return p.wcx; }
    static __device__ __forceinline__ R wcy(const ResPop<R> &p) { return p.wcy; }
};

constexpr int RES_THREADS = 512, RES_WARPS = RES_THREADS / 32;

/* V consecutive elements of a shared-memory row */
template <int V, typename T>
__device__ __forceinline__ void res_ld(const T *p, T (&v)[V])
{
    if constexpr (V == 1) v[0] = *p;
    else ldn<V>(p, v);
}
template <int V, typename T>
__device__ __forceinline__ void res_st(T *p, const T (&v)[V])
{
    if constexpr (V == 1) *p = v[0];
    else stn<V>(p, v);
}

/* Everything lives in one dynamic allocation; every function below takes its address from
 * this symbol, so that all accesses are shared-memory loads and stores. */
extern __shared__ __align__(16) unsigned char res_smem[];

__device__ __forceinline__ const ResHead &res_head() { return *reinterpret_cast<const ResHead *>(res_smem); }

/* minmod (the median of a, b and 0) on the bit patterns of FP64 values: the FP64 units are
 * the bound of these steps, the integer units are idle. The value is minmod_n's. */
__device__ __forceinline__ double res_minmod(double a, double b)
{
    const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
    const unsigned long long ma = (unsigned long long)ia & 0x7fffffffffffffffull, mb = (unsigned long long)ib & 0x7fffffffffffffffull;
    const long long m = ma < mb ? ia : ib;
    return (ia ^ ib) < 0 ? 0.0 : __longlong_as_double(m);
}
__device__ __forceinline__ float res_minmod(float a, float b) { return minmod_n(a, b, neg_part(a), neg_part(b)); }

template <int ST, bool PAIR, bool FORCE, bool CL>
struct Resident {
    using T = typename Store<ST>::T;
    using R = typename Store<ST>::R;
    using PO = ResPopOf<PAIR, R>;
    using Pop = typename PO::type;
    static constexpr int V = PAIR ? 4 : 1;
    /* a deviation survives encode and decode unchanged: the wall sums can read the planes */
    static constexpr bool EXACT = ST == 2;

    static __device__ __forceinline__ const ResRow *rows() { return reinterpret_cast<const ResRow *>(res_smem + res_head().off_rows); }
    static __device__ __forceinline__ const ResLat<R> *lats() { return reinterpret_cast<const ResLat<R> *>(res_smem + res_head().off_lat); }
    static __device__ __forceinline__ const Pop *pops(int s) { return reinterpret_cast<const Pop *>(res_smem + res_head().off_pop) + (s ? res_head().q[0] : 0); }
    static __device__ __forceinline__ T *at(uint32_t off) { return reinterpret_cast<T *>(res_smem + off); }
    static __device__ __forceinline__ int upr_of(int W) { return (W + V - 1) / V; }
    static __device__ __forceinline__ int div(int e, int n, uint32_t magic) { return n == 1 ? e : (int)__umulhi((uint32_t)e, magic); }
    /* physical plane of population a of set s */
    static __device__ __forceinline__ int phys(const ResHead &h, int s, int a, int phase)
    {
        const int M = h.q[s] + h.K[s], k = a + phase;
        return k >= M ? k - M : k;
    }
    /* byte offset of row slot `slot` of physical plane ph */
    static __device__ __forceinline__ uint32_t place(const ResHead &h, int s, int ph, int slot)
    {
        return h.off_plane[s] + ((uint32_t)(ph * h.nslot[s] + slot) * (uint32_t)h.pitch + (uint32_t)h.xoff) * (uint32_t)sizeof(T);
    }
    /* a unit of a row (rowp: its column 0), with the row's periodic images beside it where
     * the width is not a whole number of quads */
    static __device__ __forceinline__ void put(T *rowp, int x0, int W, bool images, const T (&e)[V])
    {
        if (V == 1 || !images) {
            res_st<V>(rowp + x0, e);
            return;
        }
#pragma unroll
        for (int k = 0; k < V; ++k) {
            const int x = x0 + k;
            if (x < W) rowp[x] = e[k];
            if (x < 2) rowp[x + W] = e[k];
            if (x >= W - 2 && x < W) rowp[x - W] = e[k];
        }
    }
    /* the same unit into the blocks that read the row */
    static __device__ __forceinline__ void push(const ResHead &h, int s, int ph, int rowi, int view, int x0, const T (&e)[V])
    {
        if constexpr (CL) {
            namespace cg = cooperative_groups;
            const uint16_t *to = reinterpret_cast<const uint16_t *>(res_smem + h.off_push) + 8 * rowi + 4 * view;
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const int rk = to[2 * t];
                if (rk == RES_NONE) continue;
                const ResRank &k = h.rank[rk];
                T *local = at(k.off_plane[s] + ((uint32_t)(ph * k.nslot[s] + to[2 * t + 1]) * (uint32_t)h.pitch + (uint32_t)h.xoff) * (uint32_t)sizeof(T));
                put(cg::this_cluster().map_shared_rank(local, rk), x0, h.W, V > 1 && h.xoff != 0, e);
            }
        }
    }
    static __device__ __forceinline__ R dec(T v, R winv, R rho0) { return decode<ST>(v, winv, rho0); }

    /* ---- wall rows (Sec. 3.2): one (unit, gas-bound population) per thread. rho_W from the
     * wall-bound populations as updated, before they were rounded to storage (every thread
     * of a unit forms the same sum, in population order), then f = rho_W S(u_W). ---- */
    static __device__ __forceinline__ void walls(const int (&phase)[2])
    {
        const ResHead &h = res_head();
        const int W = h.W, upr = upr_of(W);
        const int n0 = h.nwall[0] * upr, n1 = h.nwall[1] * upr;
        const int t0 = n0 * h.nh[0], total = t0 + n1 * h.nh[1];
        for (int it = threadIdx.x; it < total; it += RES_THREADS) {
            const int s = it < t0 ? 0 : 1, k0 = s ? it - t0 : it, n = s ? n1 : n0;
            const int i = k0 / n, un = k0 - i * n;
            const int r = div(un, upr, h.upr_magic), x0 = (un - r * upr) * V;   /* the wall rows come first */
            const int rowi = (s ? h.nrow[0] : 0) + r, Q = h.q[s], nh = h.nh[s];
            const ResRow rr = rows()[rowi];
            const ResLat<R> &L = lats()[rr.lat];
            const int w = (rr.flags & 2) ? 1 : 0;
            const R nsgn = w == 0 ? R(1) : R(-1), rho0 = L.rho0;
            const int ab = w == 0 ? 0 : Q - nh, a = (w == 0 ? Q - nh : 0) + i;   /* wall-bound half, this population */
            const Pop *tp = pops(s);
            R num[V];
#pragma unroll
            for (int k = 0; k < V; ++k) num[k] = R(0);
            const R *wb = reinterpret_cast<const R *>(res_smem + h.off_wall) + ((rr.wallord * h.nhmax) * upr + x0 / V) * V;
            const uint32_t pstride = (uint32_t)(h.nslot[s] * h.pitch) * (uint32_t)sizeof(T);
            uint32_t po = place(h, s, phys(h, s, ab, phase[s]), rr.own) + x0 * (uint32_t)sizeof(T);
            const uint32_t pend = h.off_plane[s] + (uint32_t)(Q + h.K[s]) * pstride, plen = (uint32_t)(Q + h.K[s]) * pstride;
#pragma unroll 6
            for (int b = 0; b < nh; ++b) {
                const Pop &p = tp[ab + b];
                const R xn = PO::cy(p) * nsgn;
                R d[V];
                if constexpr (EXACT) {
                    T raw[V];
                    res_ld<V>(at(po), raw);
#pragma unroll
                    for (int k = 0; k < V; ++k) d[k] = dec(raw[k], PO::winv(p), rho0);
                    po += pstride;
                    if (po >= pend) po -= plen;
                } else {
                    res_ld<V>(wb + b * upr * V, d);
                }
#pragma unroll
                for (int k = 0; k < V; ++k) num[k] = fma(-xn * PO::w(p), d[k], num[k]);
            }
            const R uwx = L.uw_x[w], uwy = L.uw_y[w];
            const R usw = uwx * uwx + uwy * uwy;
            const R kd = L.kdiff[s][w], kout = L.kout[s][w];
            const Pop &p = tp[a];
            const R ew = PO::cx(p) * uwx + PO::cy(p) * uwy;
            const R sm1 = ew + R(0.5) * (ew * ew - usw);    /* S / w - 1 */
            T e[V];
#pragma unroll
            for (int k = 0; k < V; ++k) {
                const R rwd = fma(rho0, kd, num[k]) / kout;   /* rho_W - rho0 */
                e[k] = encode<ST>(fma(rwd + rho0, sm1, rwd), PO::w(p), rho0);
            }
            const int ph = phys(h, s, a, phase[s]);
            put(at(place(h, s, ph, rr.own)), x0, W, V > 1 && h.xoff != 0, e);
            if (CL && (rr.flags & RES_PUSH)) push(h, s, ph, rowi, 0, x0, e);
        }
    }

    /* ---- moments in population order, and each node's collision coefficients ---- */
    static __device__ __forceinline__ void moments(const int (&phase)[2])
    {
        const ResHead &h = res_head();
        const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
        const int W = h.W, upr = upr_of(W), nc1 = (h.nunit[1] + 31) / 32, nc0 = (h.nunit[0] + 31) / 32;
        for (int u = warp; u < nc0 + nc1; u += RES_WARPS) {
            const int s = u < nc1 ? 1 : 0, nu = h.nunit[s];
            const int e = (s ? u : u - nc1) * 32 + lane;
            const bool on = e < nu;
            const int r = div(on ? e : 0, upr, h.upr_magic), x0 = ((on ? e : 0) - r * upr) * V;
            const ResRow rr = rows()[(s ? h.nrow[0] : 0) + r];
            const ResLat<R> &L = lats()[rr.lat];
            const Pop *tp = pops(s);
            const int Q = h.q[s];
            const R rho0 = L.rho0;
            const uint32_t pstride = (uint32_t)(h.nslot[s] * h.pitch) * (uint32_t)sizeof(T);
            const uint32_t plen = (uint32_t)(Q + h.K[s]) * pstride, pend = h.off_plane[s] + plen;
            uint32_t po = place(h, s, phase[s], rr.own) + x0 * (uint32_t)sizeof(T);
            R rd[V], jx[V], jy[V];
#pragma unroll
            for (int k = 0; k < V; ++k) rd[k] = jx[k] = jy[k] = R(0);
            const bool sh = on && (rr.flags & RES_SHADOW);
            R hh[3][V];
#pragma unroll
            for (int k = 0; k < V; ++k) hh[0][k] = hh[1][k] = hh[2][k] = R(0);
            auto sums = [&](const Pop &p, const T (&raw)[V], auto herm) {
                if constexpr (PAIR) {
#pragma unroll
                    for (int k = 0; k < V; k += 2) {
                        const float2 d = make_float2(dec(raw[k], p.winv2.x, rho0), dec(raw[k + 1], p.winv2.x, rho0));
                        const float2 a0 = fma2(p.w2, d, make_float2(rd[k], rd[k + 1]));
                        const float2 a1 = fma2(p.wcx2, d, make_float2(jx[k], jx[k + 1]));
                        const float2 a2 = fma2(p.wcy2, d, make_float2(jy[k], jy[k + 1]));
                        rd[k] = a0.x, rd[k + 1] = a0.y;
                        jx[k] = a1.x, jx[k + 1] = a1.y;
                        jy[k] = a2.x, jy[k + 1] = a2.y;
                        if constexpr (decltype(herm)::value) {
                            hh[0][k] = fma(p.wxx, d.x, hh[0][k]), hh[0][k + 1] = fma(p.wxx, d.y, hh[0][k + 1]);
                            hh[1][k] = fma(p.wxy, d.x, hh[1][k]), hh[1][k + 1] = fma(p.wxy, d.y, hh[1][k + 1]);
                            hh[2][k] = fma(p.wyy, d.x, hh[2][k]), hh[2][k + 1] = fma(p.wyy, d.y, hh[2][k + 1]);
                        }
                    }
                } else {
                    const R d = dec(raw[0], p.winv, rho0);
                    rd[0] = fma(p.w, d, rd[0]);
                    jx[0] = fma(p.wcx, d, jx[0]);
                    jy[0] = fma(p.wcy, d, jy[0]);
                    if constexpr (decltype(herm)::value) {
                        hh[0][0] = fma(p.wxx, d, hh[0][0]);
                        hh[1][0] = fma(p.wxy, d, hh[1][0]);
                        hh[2][0] = fma(p.wyy, d, hh[2][0]);
                    }
                }
            };
            /* quads: abscissa rows of N populations, whose planes are adjacent, all loaded before
             * the first is used (8 x 64 channel, 100 steps: 639 -> 620 us); single nodes, bound
             * by the FP64 units, one by one (the same change: 1115 -> 1141 us) */
            auto plain = [&](auto herm) {
#pragma unroll 3
                for (int a = 0; a < Q; ++a) {
                    T raw[V];
                    res_ld<V>(at(po), raw);
                    po += pstride;
                    if (po >= pend) po -= plen;
                    sums(tp[a], raw, herm);
                }
            };
            auto all = [&](auto nc, auto herm) {
                constexpr int N = decltype(nc)::value;
#pragma unroll 2
                for (int iy = 0; iy < N; ++iy) {
                    T raw[N][V];
#pragma unroll
                    for (int i = 0; i < N; ++i) res_ld<V>(at(po + (uint32_t)i * pstride), raw[i]);
                    po += N * pstride;
                    if (po >= pend) po -= plen;
#pragma unroll
                    for (int i = 0; i < N; ++i) sums(tp[iy * N + i], raw[i], herm);
                }
            };
            auto by_set = [&](auto herm) {
                if constexpr (!PAIR) plain(herm);
                else if (Q == 9) all(std::integral_constant<int, 3>{}, herm);
                else if (Q == 16) all(std::integral_constant<int, 4>{}, herm);
                else all(std::integral_constant<int, 6>{}, herm);
            };
            if (__any_sync(0xffffffffu, sh)) by_set(std::true_type{});
            else by_set(std::false_type{});
            if (!on) continue;
            /* velocity, relaxation frequency, density and (PAIR) the constant part of the
             * folded collision, as pair_node_state forms them, or the density deviation */
            R *st = reinterpret_cast<R *>(res_smem + h.off_state) + (s ? 5 * V * h.nunit[0] : 0) + V * e;
            R out[5][V];
#pragma unroll
            for (int k = 0; k < V; ++k) {
                const R rho = rho0 + rd[k];
                const R inv = R(1) / rho;
                const R ux = jx[k] * inv, uy = jy[k] * inv;
                const R tau = (L.tau_const ? L.kn_rho : L.kn_rho * inv) - L.tau_shift;
                const R om = L.dt / tau;
                out[0][k] = ux;
                out[1][k] = uy;
                out[2][k] = om;
                out[3][k] = rho;
                if constexpr (PAIR) {
                    R b = om * fma(R(-0.5) * rho, usq_of(ux, uy), rd[k]);
                    if constexpr (FORCE) b = fma(-(L.dt * rho), xi_dot(L.gx, L.gy, ux, uy), b);
                    out[4][k] = b;
                } else {
                    out[4][k] = rd[k];
                }
            }
#pragma unroll
            for (int i = 0; i < 5; ++i) res_st<V>(st + i * V * nu, out[i]);
            if (sh) {
                R *hs = reinterpret_cast<R *>(res_smem + h.off_herm) + (rr.shord * upr + x0 / V) * 6 * V;
                res_st<V>(hs, rd);
                res_st<V>(hs + V, jx);
                res_st<V>(hs + 2 * V, jy);
                res_st<V>(hs + 3 * V, hh[0]);
                res_st<V>(hs + 4 * V, hh[1]);
                res_st<V>(hs + 5 * V, hh[2]);
            }
        }
    }

    /* ---- views of shadow rows in the other set, one (unit, population) per thread ---- */
    static __device__ __forceinline__ void views(const int (&phase)[2])
    {
        const ResHead &h = res_head();
        const uint16_t *list = reinterpret_cast<const uint16_t *>(res_smem + h.off_shlist);
        const int W = h.W, upr = upr_of(W), n1 = h.nsh[1] * upr, n0 = h.nsh[0] * upr;   /* shadow units per own set */
        const int t0 = n0 * h.q[1], total = t0 + n1 * h.q[0];
        for (int i = threadIdx.x; i < total; i += RES_THREADS) {
            const int s = i < t0 ? 0 : 1;   /* the rows' own set */
            const int t = 1 - s, k0 = s == 0 ? i : i - t0, n = s == 0 ? n0 : n1;
            const int b = k0 / n, un = k0 - b * n;
            const int o = div(un, upr, h.upr_magic), x0 = (un - o * upr) * V, ord = (s == 0 ? 0 : h.nsh[0]) + o;
            const int rowi = list[ord];
            const ResRow rr = rows()[rowi];
            const R rho0 = lats()[rr.lat].rho0;
            const R *hs = reinterpret_cast<const R *>(res_smem + h.off_herm) + (ord * upr + x0 / V) * 6 * V;
            R c[6][V];
#pragma unroll
            for (int m = 0; m < 6; ++m) res_ld<V>(hs + m * V, c[m]);
            const Pop &p = pops(t)[b];
            T e[V];
#pragma unroll
            for (int k = 0; k < V; ++k) {   /* hermite_rebuild, term by term */
                R v = fma(c[1][k], PO::cx(p), c[0][k]);
                v = fma(c[2][k], PO::cy(p), v);
                v = fma(c[3][k], R(p.hxx), v);
                v = fma(c[4][k], R(p.hxy), v);
                v = fma(c[5][k], R(p.hyy), v);
                e[k] = encode<ST>(v, PO::w(p), rho0);
            }
            const int ph = phys(h, t, b, phase[t]);
            if (rr.view != RES_NONE) put(at(place(h, t, ph, rr.view)), x0, W, V > 1 && h.xoff != 0, e);
            if (CL && (rr.flags & RES_PUSH)) push(h, t, ph, rowi, 1, x0, e);
        }
    }

    /* ---- one round of the update of set s: abscissa rows iy [lo, hi) of the product rule,
     * an item being a unit x rpg of those rows (n populations each, so that the sign of
     * xi_x is the same in every lane); warps take 32 items at a time, starting at u0 ---- */
    static __device__ __forceinline__ void update(int s, int lo, int hi, int phase, int u0, uint32_t step_key, bool sr)
    {
        const ResHead &h = res_head();
        const int lane = threadIdx.x & 31, nu = h.nunit[s], rpg = h.rpg[s], n = h.n[s];
        const int items = nu * ((hi - lo + rpg - 1) / rpg), nunits = (items + 31) / 32;
        const int W = h.W, upr = upr_of(W), r0 = s ? h.nrow[0] : 0;
        const bool images = V > 1 && h.xoff != 0;
        const uint32_t pitchb = (uint32_t)h.pitch * (uint32_t)sizeof(T), pstride = (uint32_t)h.nslot[s] * pitchb;
        const uint32_t umagic = h.unit_magic[s], upmagic = h.upr_magic;
        const uint32_t base = h.off_plane[s] + (uint32_t)h.xoff * (uint32_t)sizeof(T);
        const int M = h.q[s] + h.K[s], K = h.K[s];
        const R *stb = reinterpret_cast<const R *>(res_smem + h.off_state) + (s ? 5 * V * h.nunit[0] : 0);
        const Pop *tp = pops(s);
        for (int u = u0; u < nunits; u += RES_WARPS) {
            const int item = u * 32 + lane;
            if (item >= items) continue;
            const int g = div(item, nu, umagic), e = item - g * nu;
            const int r = div(e, upr, upmagic), x0 = (e - r * upr) * V;
            const ResRow rr = rows()[r0 + r];
            const ResLat<R> &L = lats()[rr.lat];
            const R rho0 = L.rho0;
            R stt[5][V];
#pragma unroll
            for (int i = 0; i < 5; ++i) res_ld<V>(stb + i * V * nu + V * e, stt[i]);
            R gx = R(0), gy = R(0), dtl = R(0);
            if constexpr (FORCE) {
                gx = L.gx;
                gy = L.gy;
                dtl = L.dt;
            }
            /* byte offsets, relative to a plane, of the unit and of its y neighbours; the x
             * neighbours relative to the unit: the row's other end where the width is a
             * whole number of units, the images beside the row else */
            const uint32_t xb = (uint32_t)x0 * (uint32_t)sizeof(T);
            const uint32_t oo = rr.own * pitchb + xb;
            const uint32_t m2 = rr.m2 * pitchb + xb, m1 = rr.m1 * pitchb + xb, p1 = rr.p1 * pitchb + xb, p2 = rr.p2 * pitchb + xb;
            int ox[4] = {0, 0, 0, 0};
            if constexpr (PAIR) {
                ox[0] = (!images && x0 == 0) ? W - 2 : -2;
                ox[1] = (!images && x0 + 4 == W) ? 4 - W : 4;
            } else {
                ox[0] = x0 >= 2 ? -2 : W - 2;
                ox[1] = x0 >= 1 ? -1 : W - 1;
                ox[2] = x0 + 1 < W ? 1 : 1 - W;
                ox[3] = x0 + 2 < W ? 2 : 2 - W;
            }
            const bool special = (rr.flags & (3 | RES_PUSH)) != 0;
            const R wsgn = (rr.flags & 1) ? R(1) : ((rr.flags & 2) ? R(-1) : R(0));
            const int iy1 = min(hi, lo + (g + 1) * rpg);
            for (int iy = lo + g * rpg; iy < iy1; ++iy) {
                const int a0 = iy * n;
                int ph = a0 + phase;
                ph = ph >= M ? ph - M : ph;
                int pn = ph - K;
                pn = pn < 0 ? pn + M : pn;
                const uint32_t pa = base + (uint32_t)ph * pstride, pw = base + (uint32_t)pn * pstride;
                const Pop *ta = tp + a0;
                const R cy = PO::cy(*ta);
                /* the window rows j - 2s, j - s, j + s, s = sign(xi_y) */
                const bool up = cy > R(0);
                const uint32_t w0 = up ? m2 : p2, w1 = up ? m1 : p1, w3 = up ? p1 : m1;
                /* what follows a population's update on wall rows (the unrounded wall-bound
                 * value is kept) and on rows other blocks read */
                auto finish = [&](int a, const R (&dn)[V], const T (&ev)[V], uint32_t dst) {
                    put(at(dst - xb), x0, W, images, ev);
                    if (special) {
                        if (!EXACT && cy * wsgn < R(0)) {
                            const int i = (rr.flags & 2) ? a - (h.q[s] - h.nh[s]) : a;
                            res_st<V>(reinterpret_cast<R *>(res_smem + h.off_wall) + ((rr.wallord * h.nhmax + i) * upr + x0 / V) * V, dn);
                        }
                        if (CL && (rr.flags & RES_PUSH)) {
                            int k = a + phase - K;   /* physical plane written */
                            k = k < 0 ? k + M : (k >= M ? k - M : k);
                            push(h, s, k, r0 + r, 0, x0, ev);
                        }
                    }
                };
                if constexpr (PAIR) {
                    const RingPop &pr = *ta;
                    const float2 cy2 = pr.cy2, nacy2 = pr.nacy2, ky2 = pr.ky2;
                    const bool hy = nacy2.x != 0.0f;
                    float2 ux[2], uy[2], om[2], P[2], B[2], dr[2];
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        ux[k] = make_float2(stt[0][2 * k], stt[0][2 * k + 1]);
                        uy[k] = make_float2(stt[1][2 * k], stt[1][2 * k + 1]);
                        om[k] = make_float2(-stt[2][2 * k], -stt[2][2 * k + 1]);
                        P[k] = make_float2(stt[2][2 * k] * stt[3][2 * k], stt[2][2 * k + 1] * stt[3][2 * k + 1]);
                        B[k] = make_float2(stt[4][2 * k], stt[4][2 * k + 1]);
                        if constexpr (FORCE) dr[k] = make_float2(dtl * stt[3][2 * k], dtl * stt[3][2 * k + 1]);
                    }
                    const float2 nrho02 = f2(-rho0);
                    auto pop = [&](int ix, auto sxc) {
                        constexpr int SX = decltype(sxc)::value;
                        const RingPop &px = tp[ix];   /* the abscissa's constants: the same in every lane */
                        const uint32_t src = pa + (uint32_t)ix * pstride;
                        float2 w2 = f2(1.0f), winv2 = f2(1.0f);
                        if constexpr (ST == 1) {
                            w2 = ta[ix].w2;
                            winv2 = ta[ix].winv2;
                        }
                        auto dec2 = [&](T a, T b) -> float2 {
                            const float2 raw = make_float2(to_r(a), to_r(b));
                            if constexpr (ST == 1) return fma2(raw, winv2, nrho02);
                            else return raw;
                        };
                        T own[4];
                        ldn<4>(at(src + oo), own);
                        float2 v[2], c[2];
#pragma unroll
                        for (int k = 0; k < 2; ++k) v[k] = dec2(own[2 * k], own[2 * k + 1]);
#pragma unroll
                        for (int k = 0; k < 2; ++k) {
                            float2 eu;
                            if constexpr (SX == 0) eu = mul2(cy2, uy[k]);
                            else eu = fma2(cy2, uy[k], mul2(px.cx2, ux[k]));
                            const float2 t = fma2(mul2(f2(0.5f), eu), eu, eu);
                            c[k] = fma2(om[k], v[k], fma2(P[k], t, B[k]));
                            if constexpr (FORCE) {
                                const float2 gxi2 = f2(xi_dot(px.cx2.x, cy2.x, gx, gy));
                                c[k] = fma2(dr[k], fma2(gxi2, eu, gxi2), c[k]);
                            }
                        }
                        if constexpr (SX != 0) {
                            T hl[2], hr[2];
                            ld2(at(src + oo) + ox[0], hl);
                            ld2(at(src + oo) + ox[1], hr);
                            const float2 hl2 = dec2(hl[0], hl[1]), hr2 = dec2(hr[0], hr[1]);
                            const float kx = px.kx;
                            float D[4];
                            float d[6], nn[6], m[5];
                            if constexpr (SX > 0) {
                                d[0] = hl2.y - hl2.x;
                                d[1] = v[0].x - hl2.y;
                                d[2] = v[0].y - v[0].x;
                                d[3] = v[1].x - v[0].y;
                                d[4] = v[1].y - v[1].x;
                                d[5] = hr2.x - v[1].y;
                            } else {
                                d[0] = v[0].x - hl2.y;
                                d[1] = v[0].y - v[0].x;
                                d[2] = v[1].x - v[0].y;
                                d[3] = v[1].y - v[1].x;
                                d[4] = hr2.x - v[1].y;
                                d[5] = hr2.y - hr2.x;
                            }
#pragma unroll
                            for (int i = 0; i < 6; ++i) nn[i] = neg_part(d[i]);
#pragma unroll
                            for (int i = 0; i < 5; ++i) m[i] = minmod_n(d[i], d[i + 1], nn[i], nn[i + 1]);
#pragma unroll
                            for (int k = 0; k < 4; ++k) D[k] = fmaf(SX > 0 ? kx : -kx, m[k + 1] - m[k], d[k + 1]);
                            c[0] = fma2(px.ncx2, make_float2(D[0], D[1]), c[0]);
                            c[1] = fma2(px.ncx2, make_float2(D[2], D[3]), c[1]);
                        }
                        if (hy) {
                            T y0[4], y1[4], y3[4];
                            ldn<4>(at(src + w0), y0);
                            ldn<4>(at(src + w1), y1);
                            ldn<4>(at(src + w3), y3);
#pragma unroll
                            for (int k = 0; k < 2; ++k) {
                                const float2 b0 = dec2(y0[2 * k], y0[2 * k + 1]), b1 = dec2(y1[2 * k], y1[2 * k + 1]);
                                const float2 b3 = dec2(y3[2 * k], y3[2 * k + 1]);
                                const float2 d0 = sub2(b1, b0), d1 = sub2(v[k], b1), d2 = sub2(b3, v[k]);
                                float2 ma, mb;
                                {
                                    const float l = fminf(d1.x, 0.0f), u2 = fmaxf(d1.x, 0.0f);
                                    ma.x = fminf(fmaxf(d0.x, l), u2);
                                    mb.x = fminf(fmaxf(d2.x, l), u2);
                                }
                                {
                                    const float l = fminf(d1.y, 0.0f), u2 = fmaxf(d1.y, 0.0f);
                                    ma.y = fminf(fmaxf(d0.y, l), u2);
                                    mb.y = fminf(fmaxf(d2.y, l), u2);
                                }
                                c[k] = fma2(nacy2, fma2(ky2, sub2(mb, ma), d1), c[k]);
                            }
                        }
                        const float2 dn0 = add2(v[0], c[0]), dn1 = add2(v[1], c[1]);
                        float2 e0 = dn0, e1 = dn1;
                        if constexpr (ST == 1) {
                            e0 = mul2(w2, add2(f2(rho0), dn0));
                            e1 = mul2(w2, add2(f2(rho0), dn1));
                        }
                        const uint32_t dst = pw + (uint32_t)ix * pstride + oo;
                        if (!special && !images) {
                            pair_st<ST>(at(dst), e0, e1);
                        } else {
                            const T ev[4] = {from_r<T>(e0.x), from_r<T>(e0.y), from_r<T>(e1.x), from_r<T>(e1.y)};
                            const R dn[4] = {dn0.x, dn0.y, dn1.x, dn1.y};
                            finish(a0 + ix, dn, ev, dst);
                        }
                    };
                    int ix = 0;
#pragma unroll 1
                    for (; ix < n / 2; ++ix) pop(ix, std::integral_constant<int, -1>{});
                    if (n & 1) {
                        pop(ix, std::integral_constant<int, 0>{});
                        ++ix;
                    }
#pragma unroll 1
                    for (; ix < n; ++ix) pop(ix, std::integral_constant<int, 1>{});
                } else {
                    const R ux = stt[0][0], uy = stt[1][0], om = stt[2][0], rho = stt[3][0], rhod = stt[4][0];
                    const R usq = usq_of(ux, uy);
                    R gu = R(0), dtr = R(0);
                    if constexpr (FORCE) {
                        gu = xi_dot(gx, gy, ux, uy);
                        dtr = dtl * rho;
                    }
                    const R cry = ta->cry, ky = ta->ky;
                    /* the window runs from upwind for either sign: for xi_y < 0 every difference,
                     * and so the flux difference, is the printed one with its sign changed */
                    const R nacry = up ? -cry : cry;
                    const bool hy = cry != R(0);
#pragma unroll 1
                    for (int ix = 0; ix < n; ++ix) {
                        const uint32_t src = pa + (uint32_t)ix * pstride;
                        const Pop &px = tp[ix];
                        const R w = ta[ix].w, winv = ta[ix].winv, cx = px.cx, crx = px.crx;
                        const T *c0 = at(src + oo);
                        const R v = dec(*c0, winv, rho0);
                        const R eu = xi_dot(cx, cy, ux, uy);
                        R inc = om * (deq(rhod, rho, eu, usq) - v);
                        if (crx != R(0)) {
                            R d0, d1, d2, kf;
                            const R l1 = dec(c0[ox[1]], winv, rho0), q0 = dec(c0[ox[2]], winv, rho0);
                            R far;
                            if (crx > R(0)) {
                                far = dec(c0[ox[0]], winv, rho0);
                                d0 = l1 - far;
                                d1 = v - l1;
                                d2 = q0 - v;
                                kf = px.kx;
                            } else {
                                far = dec(c0[ox[3]], winv, rho0);
                                d0 = v - l1;
                                d1 = q0 - v;
                                d2 = far - q0;
                                kf = -px.kx;
                            }
                            inc = fma(-crx, fma(kf, res_minmod(d1, d2) - res_minmod(d0, d1), d1), inc);
                        }
                        if (hy) {
                            const R b0 = dec(*at(src + w0), winv, rho0), b1 = dec(*at(src + w1), winv, rho0);
                            const R b3 = dec(*at(src + w3), winv, rho0);
                            const R d0 = b1 - b0, d1 = v - b1, d2 = b3 - v;
                            inc = fma(nacry, fma(ky, res_minmod(d1, d2) - res_minmod(d0, d1), d1), inc);
                        }
                        if constexpr (FORCE) inc = force_inc(dtr, xi_dot(cx, cy, gx, gy), eu, gu, inc);
                        const R dn = v + inc;
                        T ev[1];
                        if (sr) ev[0] = encode_sr<ST>(dn, w, rho0, sr_bits(x0, (int)rr.j, W, a0 + ix, step_key));
                        else ev[0] = encode<ST>(dn, w, rho0);
                        const uint32_t dst = pw + (uint32_t)ix * pstride + oo;
                        if (!special) {
                            *at(dst) = ev[0];
                        } else {
                            const R dna[1] = {dn};
                            finish(a0 + ix, dna, ev, dst);
                        }
                    }
                }
            }
        }
    }
};

/* nparts parts of one lattice each on one block of a cluster (CL), or bundles of lattices,
 * one block at a time, from a queue. par [lattice][2]: launch parameters from the level
 * `base` (see launch_ring_batch); osc: wall values of every step (n > 0) of a lattice with
 * oscillating walls. advance = 0: nothing is written back. */
template <int ST, bool PAIR, bool FORCE, bool CL>
__global__ void __launch_bounds__(RES_THREADS, 1)
    resident_kernel(const unsigned char *__restrict__ plan, const uint32_t *__restrict__ part_off, int nparts,
                    const StepParams<typename Store<ST>::R> *__restrict__ par2, const RingTab *__restrict__ tabs,
                    int nsteps, int base, uint32_t step0, int advance, unsigned int *queue,
                    const __grid_constant__ ResOsc<typename Store<ST>::R> osc)
{
    using RT = Resident<ST, PAIR, FORCE, CL>;
    using T = typename RT::T;
    using R = typename RT::R;
    namespace cg = cooperative_groups;
    const ResHead &h = res_head();
    __shared__ int part_sh;
    const int tid = threadIdx.x;
    for (;;) {
        int part;
        if constexpr (CL) {
            part = (int)cg::this_cluster().block_rank();
        } else {
            __syncthreads();
            if (tid == 0) part_sh = (int)atomicAdd(queue, 1u);
            __syncthreads();
            part = part_sh;
            if (part >= nparts) return;
        }
        /* tables */
        const unsigned char *pp = plan + part_off[part];
        const ResHead *gh = reinterpret_cast<const ResHead *>(pp);
        const int table = gh->table_bytes;   /* the part kept in shared memory, then the rows' global places */
        for (int k = tid; k < table / 16; k += RES_THREADS)
            reinterpret_cast<uint4 *>(res_smem)[k] = reinterpret_cast<const uint4 *>(pp)[k];
        if constexpr (CL) cg::this_cluster().sync();   /* every block is running: its memory may be stored into */
        else __syncthreads();
        const ResGRow *grow = reinterpret_cast<const ResGRow *>(pp + h.off_grow);
        const int nlat = h.nlat;
        /* level read: parameters [lat][base]; level written: that of an even or odd count */
        const int sel = nsteps & 1 ? base : base ^ 1;
        ResLat<R> *lats = reinterpret_cast<ResLat<R> *>(res_smem + h.off_lat);
        const int *ids = reinterpret_cast<const int *>(res_smem + h.off_ids);
        for (int k = tid; k < nlat; k += RES_THREADS) {
            const StepParams<R> &p = par2[2 * (size_t)ids[k] + base];
            ResLat<R> L;
            L.rho0 = p.rho0;
            L.dt = p.dt;
            L.kn_rho = p.kn_rho;
            L.tau_shift = p.tau_shift;
            L.tau_const = p.tau_const;
            L.gx = p.gx;
            L.gy = p.gy;
            for (int w = 0; w < 2; ++w) {
                L.uw_x[w] = p.uw_x[w];
                L.uw_y[w] = p.uw_y[w];
                for (int s = 0; s < 2; ++s) {
                    L.kdiff[s][w] = p.kdiff[s][w];
                    L.kout[s][w] = p.kout[s][w];
                }
            }
            lats[k] = L;
        }
        typename RT::Pop *pops = reinterpret_cast<typename RT::Pop *>(res_smem + h.off_pop);
        if constexpr (PAIR) {
            constexpr int NW = (int)(sizeof(RingPop) / 16);
            for (int k = tid; k < (h.q[0] + h.q[1]) * NW; k += RES_THREADS) {
                const int i = k / NW, s = i < h.q[0] ? 0 : 1;
                reinterpret_cast<uint4 *>(pops)[k] = reinterpret_cast<const uint4 *>(&tabs[ids[0]].pop[s][s ? i - h.q[0] : i])[k - i * NW];
            }
        } else {
            const StepParams<R> &p = par2[2 * (size_t)ids[0] + base];
            for (int k = tid; k < h.q[0] + h.q[1]; k += RES_THREADS) {
                const SetConst<R> &c = p.set[k < h.q[0] ? 0 : 1];
                const int a = k < h.q[0] ? k : k - h.q[0];
                pops[k] = ResPop<R>{c.cx[a], c.cy[a], c.crx[a], c.cry[a], c.kx[a], c.ky[a], c.w[a], c.winv[a],
                                    c.wcx[a], c.wcy[a], c.wxx[a], c.wxy[a], c.wyy[a], c.hxx[a], c.hxy[a], c.hyy[a]};
            }
        }
        /* own populations of the level read */
        const int W = h.W;
        int phase[2] = {0, 0};
        for (int s = 0; s < 2; ++s) {
            const int nr = h.nrow[s], q = h.q[s], r0 = s ? h.nrow[0] : 0;
            const int per = nr * W, total = q * per;
            for (int k = tid; k < total; k += RES_THREADS) {
                const int a = k / per, i = k - a * per, r = i / W, x = i - r * W;
                const ResGRow g = grow[r0 + r];
                const StepParams<R> &p = par2[2 * (size_t)g.lat + base];
                const T v = static_cast<const T *>(p.fin[s])[(size_t)a * p.plane + (size_t)g.j * p.pitch + x + LB_GHOST];
                const ResRow rr = RT::rows()[r0 + r];
                T *row = RT::at(RT::place(h, s, a, rr.own));
                row[x] = v;
                if (h.xoff != 0) {
                    if (x < 2) row[x + W] = v;
                    if (x >= W - 2) row[x - W] = v;
                }
                if constexpr (CL) {
                    if (rr.flags & RES_PUSH) {
                        const uint16_t *to = reinterpret_cast<const uint16_t *>(res_smem + h.off_push) + 8 * (r0 + r);
                        for (int t = 0; t < 2; ++t) {
                            const int rk = to[2 * t];
                            if (rk == RES_NONE) continue;
                            const ResRank &kk = h.rank[rk];
                            T *local = RT::at(kk.off_plane[s] + ((uint32_t)(a * kk.nslot[s] + to[2 * t + 1]) * (uint32_t)h.pitch + (uint32_t)h.xoff) * (uint32_t)sizeof(T));
                            T *rrow = cg::this_cluster().map_shared_rank(local, rk);
                            rrow[x] = v;
                            if (h.xoff != 0) {
                                if (x < 2) rrow[x + W] = v;
                                if (x >= W - 2) rrow[x - W] = v;
                            }
                        }
                    }
                }
            }
        }
        __syncthreads();
        const bool sr = !PAIR && h.sr != 0;
        const int warp = tid / 32, nwall = h.nwall[0] + h.nwall[1], nsh = h.nsh[0] + h.nsh[1];
        for (int st = 0;; ++st) {
            if (st > 0 && nwall > 0) {
                RT::walls(phase);
                __syncthreads();
            }
            RT::moments(phase);
            __syncthreads();
            if (st == nsteps) break;
            if (nsh > 0) RT::views(phase);
            if constexpr (CL) cg::this_cluster().sync();
            else if (nsh > 0) __syncthreads();
            for (int rd = 0; rd < h.rounds; ++rd) {
                /* set 1 first: its items are the longer ones; the warps go on in set 0 where
                 * set 1 left off */
                const int kr1 = h.kr[1], kr0 = h.kr[0];
                const int lo1 = min(h.n[1], rd * kr1), hi1 = min(h.n[1], lo1 + kr1);
                const int lo0 = min(h.n[0], rd * kr0), hi0 = min(h.n[0], lo0 + kr0);
                const int units1 = (h.nunit[1] * ((hi1 - lo1 + h.rpg[1] - 1) / h.rpg[1]) + 31) / 32;
                RT::update(1, lo1, hi1, phase[1], warp, step0 + (uint32_t)st + 1u, sr);
                RT::update(0, lo0, hi0, phase[0], (warp + RES_WARPS - units1 % RES_WARPS) % RES_WARPS, step0 + (uint32_t)st + 1u, sr);
                if (rd + 1 < h.rounds) {
                    if constexpr (CL) cg::this_cluster().sync();
                    else __syncthreads();
                }
            }
            for (int s = 0; s < 2; ++s) {
                phase[s] -= h.K[s];
                if (phase[s] < 0) phase[s] += h.q[s] + h.K[s];
            }
            if (osc.n > 0 && tid < 2) {   /* oscillating walls: the new level's values */
                const int w = tid;
                lats[0].uw_x[w] = osc.v[st][w][0];
                lats[0].uw_y[w] = osc.v[st][w][1];
                for (int s = 0; s < 2; ++s) {
                    lats[0].kdiff[s][w] = osc.v[st][w][2 + s];
                    lats[0].kout[s][w] = osc.v[st][w][4 + s];
                }
            }
            __syncthreads();
        }
        if constexpr (CL) cg::this_cluster().sync();   /* no block leaves while another may still store into it */
        else __syncthreads();
        if (advance) {
            for (int s = 0; s < 2; ++s) {
                const int nr = h.nrow[s], r0 = s ? h.nrow[0] : 0;
                for (int view = 0; view < 2; ++view) {
                    const int t = view ? 1 - s : s;   /* the set the values are in */
                    const int q = h.q[t], per = nr * W, total = q * per;
                    for (int k = tid; k < total; k += RES_THREADS) {
                        const int a = k / per, i = k - a * per, r = i / W, x = i - r * W;
                        const ResRow rr = RT::rows()[r0 + r];
                        if (view && !(rr.flags & RES_SHADOW)) continue;
                        const ResGRow g = grow[r0 + r];
                        const StepParams<R> &p = par2[2 * (size_t)g.lat + sel];
                        T v;
                        if (!view) {
                            v = RT::at(RT::place(h, t, RT::phys(h, t, a, phase[t]), rr.own))[x];
                        } else {   /* as views() forms it */
                            const R *hs = reinterpret_cast<const R *>(res_smem + h.off_herm) +
                                          (rr.shord * RT::upr_of(W) + x / RT::V) * 6 * RT::V + x % RT::V;
                            const typename RT::Pop &pc = RT::pops(t)[a];
                            using PO = typename RT::PO;
                            R d = fma(hs[RT::V], PO::cx(pc), hs[0]);
                            d = fma(hs[2 * RT::V], PO::cy(pc), d);
                            d = fma(hs[3 * RT::V], R(pc.hxx), d);
                            d = fma(hs[4 * RT::V], R(pc.hxy), d);
                            d = fma(hs[5 * RT::V], R(pc.hyy), d);
                            v = encode<ST>(d, PO::w(pc), lats[rr.lat].rho0);
                        }
                        put1r(p, static_cast<T *>(p.fout[t]) + (size_t)a * p.plane + (size_t)g.j * p.pitch, x, g.j, v);
                    }
                }
            }
            /* carried moments, summed in population order */
            for (int s = 0; s < 2; ++s) {
                const int nr = h.nrow[s], r0 = s ? h.nrow[0] : 0, q = h.q[s];
                for (int k = tid; k < nr * W; k += RES_THREADS) {
                    const int r = k / W, x = k - r * W;
                    const ResGRow g = grow[r0 + r];
                    const StepParams<R> &p = par2[2 * (size_t)g.lat + sel];
                    R *aout = static_cast<R *>(p.aux_out);
                    if (!aout) continue;
                    const R rho0 = p.rho0;
                    R rd = R(0), jx = R(0), jy = R(0);
                    const int own = RT::rows()[r0 + r].own;
                    for (int a = 0; a < q; ++a) {
                        const typename RT::Pop &pc = RT::pops(s)[a];
                        using PO = typename RT::PO;
                        const R d = decode<ST>(RT::at(RT::place(h, s, RT::phys(h, s, a, phase[s]), own))[x], PO::winv(pc), rho0);
                        rd = fma(PO::w(pc), d, rd);
                        jx = fma(PO::wcx(pc), d, jx);
                        jy = fma(PO::wcy(pc), d, jy);
                    }
                    const size_t ap = (size_t)p.pitch * p.ny, m = (size_t)g.j * p.pitch + x;
                    aout[m] = rd;
                    aout[ap + m] = jx;
                    aout[2 * ap + m] = jy;
                }
            }
        }
        if constexpr (CL) return;
    }
}

template <int ST, bool PAIR, bool FORCE, bool CL>
int resident_launch(const ResLaunch &a)
{
    using R = typename Store<ST>::R;
    static_assert(sizeof(ResLat<R>) <= 24 * sizeof(R), "room of a lattice in the plan");
    auto kern = resident_kernel<ST, PAIR, FORCE, CL>;
    /* The shared-memory limit (and leave for clusters beyond the portable size) is the
     * kernel's, on a device, for every context and host thread: set once, to the most any plan
     * takes. (Set to the plan's own size on each launch, one thread lowered it between
     * another's call and launch.) */
    static std::atomic<bool> ready[64];
    int dev = 0;
    cudaGetDevice(&dev);
    dev &= 63;
    if (!ready[dev].load(std::memory_order_acquire)) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)res_smem_limit(CL)) != cudaSuccess ||
            (CL && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)) {
            cudaGetLastError();
            return -1;
        }
        ready[dev].store(true, std::memory_order_release);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(RES_THREADS);
    cfg.dynamicSmemBytes = a.plan->smem;
    cfg.stream = static_cast<cudaStream_t>(a.stream);
    cudaLaunchAttribute at[1];
    if constexpr (CL) {
        cfg.gridDim = dim3(a.plan->cluster);
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = a.plan->cluster;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
    }
    if (a.query) {
        int n = 0;
        cudaError_t e;
        if constexpr (CL) e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
        else e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, RES_THREADS, a.plan->smem);
        if (e != cudaSuccess) cudaGetLastError();
        return e == cudaSuccess && n > 0 ? 0 : -1;
    }
    if constexpr (!CL) {
        cfg.gridDim = dim3(a.plan->parts < a.blocks ? a.plan->parts : a.blocks);
        if (cudaMemsetAsync(a.queue, 0, sizeof(unsigned int), cfg.stream) != cudaSuccess) return -1;
    }
    const ResOsc<R> &osc = *static_cast<const ResOsc<R> *>(a.osc);
    const unsigned char *plan = static_cast<const unsigned char *>(a.d_plan);
    const StepParams<R> *par = static_cast<const StepParams<R> *>(a.params);
    return cudaLaunchKernelEx(&cfg, kern, plan, a.d_off, a.plan->parts, par, a.tabs, a.nsteps, a.base, a.step0, a.advance,
                              a.queue, osc) == cudaSuccess
               ? 0
               : -1;
}

template <int ST, bool PAIR>
int launch_resident_store(const ResLaunch &a)
{
    if (a.plan->cluster > 1)
        return a.force ? resident_launch<ST, PAIR, true, true>(a) : resident_launch<ST, PAIR, false, true>(a);
    return a.force ? resident_launch<ST, PAIR, true, false>(a) : resident_launch<ST, PAIR, false, false>(a);
}

}  // namespace lbk
