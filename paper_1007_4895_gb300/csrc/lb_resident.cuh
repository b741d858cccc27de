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

template <int ST, bool PAIR, bool FORCE, bool CL>
struct Resident {
    using T = typename Store<ST>::T;
    using R = typename Store<ST>::R;
    using PO = ResPopOf<PAIR, R>;
    using Pop = typename PO::type;
    static constexpr int V = PAIR ? 4 : 1;
    /* a deviation survives encode and decode unchanged: the wall sums can read the planes */
    static constexpr bool EXACT = ST == 2;

    const ResHead &h;
    unsigned char *sm;
    const ResRow *rows;
    const ResLat<R> *lats;
    const Pop *pops;   /* [2][LB_QMAX] */
    int warp, lane, W, upr, pitch, xoff;
    uint32_t rowb;

    __device__ __forceinline__ Resident(const ResHead &hh, unsigned char *s)
        : h(hh), sm(s), rows(reinterpret_cast<const ResRow *>(s + hh.off_rows)),
          lats(reinterpret_cast<const ResLat<R> *>(s + hh.off_lat)), pops(reinterpret_cast<const Pop *>(s + hh.off_pop)),
          warp(threadIdx.x / 32), lane(threadIdx.x & 31), W(hh.W), upr((hh.W + V - 1) / V), pitch(hh.pitch),
          xoff(hh.xoff), rowb(hh.pitch * sizeof(T))
    {
    }
    __device__ __forceinline__ int phys(int s, int a, int phase) const
    {
        const int M = h.q[s] + h.K[s];
        int k = a + phase;
        return k >= M ? k - M : k;
    }
    __device__ __forceinline__ T *plane(int s, int ph) const
    {
        return reinterpret_cast<T *>(sm + h.off_plane[s] + (uint32_t)ph * h.nslot[s] * rowb);
    }
    /* unit e of set s: row and first column */
    __device__ __forceinline__ void locate(int e, int &r, int &x0) const
    {
        r = upr == 1 ? e : (int)__umulhi((uint32_t)e, h.upr_magic);
        x0 = (e - r * upr) * V;
    }
    __device__ __forceinline__ R *state(int s) const
    {
        return reinterpret_cast<R *>(sm + h.off_state) + (s ? 5 * V * h.nunit[0] : 0);
    }
    /* the row's periodic images beside it (only rows whose width is not a whole number of
     * quads keep any), then the copies in other blocks */
    __device__ __forceinline__ void put(T *pl, int slot, int x0, const T (&e)[V]) const
    {
        T *row = pl + slot * pitch + xoff;
        if (V == 1 || xoff == 0 || x0 + V <= W) {
            res_st<V>(row + x0, e);
        } else {
#pragma unroll
            for (int k = 0; k < V; ++k)
                if (x0 + k < W) row[x0 + k] = e[k];
        }
        if (V > 1 && xoff != 0) {
#pragma unroll
            for (int k = 0; k < V; ++k) {
                const int x = x0 + k;
                if (x < 2) row[x + W] = e[k];
                if (x >= W - 2 && x < W) row[x - W] = e[k];
            }
        }
    }
    __device__ __forceinline__ void push(int s, int ph, const uint16_t *to, int x0, const T (&e)[V]) const
    {
        namespace cg = cooperative_groups;
        if constexpr (CL) {
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const int rk = to[2 * t];
                if (rk == RES_NONE) continue;
                const ResRank &k = h.rank[rk];
                T *local = reinterpret_cast<T *>(sm + k.off_plane[s] + (uint32_t)ph * k.nslot[s] * rowb);
                put(cg::this_cluster().map_shared_rank(local, rk), to[2 * t + 1], x0, e);
            }
        }
    }
    __device__ __forceinline__ const uint16_t *pushes(int row, int view) const
    {
        return reinterpret_cast<const uint16_t *>(sm + h.off_push) + 8 * row + 4 * view;
    }
    static __device__ __forceinline__ R dec(T v, R winv, R rho0) { return decode<ST>(v, winv, rho0); }

    /* ---- 1. moments and collision coefficients (and the wall fill of wall rows) ---- */
    template <bool FILL>
    __device__ void moments(const int (&phase)[2])
    {
        const int nc[2] = {(h.nunit[0] + 31) / 32, (h.nunit[1] + 31) / 32};
        for (int u = warp; u < nc[0] + nc[1]; u += RES_WARPS) {
            const int s = u < nc[1] ? 1 : 0;
            const int e = (s ? u : u - nc[1]) * 32 + lane;
            const bool on = e < h.nunit[s];
            int r, x0;
            locate(on ? e : 0, r, x0);
            const int rowi = (s ? h.nrow[0] : 0) + r;
            const ResRow rr = rows[rowi];
            const ResLat<R> &L = lats[rr.lat];
            const Pop *tp = pops + s * LB_QMAX;
            const int Q = h.q[s];
            const R rho0 = L.rho0;
            const int off = rr.own * pitch + xoff + x0;
            const bool wall = on && (rr.flags & 3);
            if (FILL && wall) wall_fill(s, rr, rowi, x0, phase[s], L);
            R rd[V], jx[V], jy[V], hh[3][V];
#pragma unroll
            for (int k = 0; k < V; ++k) rd[k] = jx[k] = jy[k] = hh[0][k] = hh[1][k] = hh[2][k] = R(0);
            const bool sh = on && (rr.flags & RES_SHADOW);
            const int M = Q + h.K[s];
            int ph = phase[s];
            if (__any_sync(0xffffffffu, sh)) {
#pragma unroll 4
                for (int a = 0; a < Q; ++a) {
                    T raw[V];
                    res_ld<V>(plane(s, ph) + off, raw);
                    ph = ph + 1 == M ? 0 : ph + 1;
                    const Pop &p = tp[a];
#pragma unroll
                    for (int k = 0; k < V; ++k) {
                        const R d = dec(raw[k], PO::winv(p), rho0);
                        rd[k] = fma(PO::w(p), d, rd[k]);
                        jx[k] = fma(PO::wcx(p), d, jx[k]);
                        jy[k] = fma(PO::wcy(p), d, jy[k]);
                        hh[0][k] = fma(R(p.wxx), d, hh[0][k]);
                        hh[1][k] = fma(R(p.wxy), d, hh[1][k]);
                        hh[2][k] = fma(R(p.wyy), d, hh[2][k]);
                    }
                }
            } else {
#pragma unroll 6
                for (int a = 0; a < Q; ++a) {
                    T raw[V];
                    res_ld<V>(plane(s, ph) + off, raw);
                    ph = ph + 1 == M ? 0 : ph + 1;
                    const Pop &p = tp[a];
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
                        }
                    } else {
                        const R d = dec(raw[0], PO::winv(p), rho0);
                        rd[0] = fma(PO::w(p), d, rd[0]);
                        jx[0] = fma(PO::wcx(p), d, jx[0]);
                        jy[0] = fma(PO::wcy(p), d, jy[0]);
                    }
                }
            }
            if (!on) continue;
            /* velocity, relaxation frequency, and (PAIR) the constant part of the folded
             * collision, as pair_node_state forms them, or the density deviation */
            R *st = state(s) + V * e;
            const int n = V * h.nunit[s];
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
            for (int i = 0; i < 5; ++i) res_st<V>(st + i * n, out[i]);
            if (sh) {
                R *hs = reinterpret_cast<R *>(sm + h.off_herm) + ((size_t)rr.shord * upr + x0 / V) * 6 * V;
                res_st<V>(hs, rd);
                res_st<V>(hs + V, jx);
                res_st<V>(hs + 2 * V, jy);
                res_st<V>(hs + 3 * V, hh[0]);
                res_st<V>(hs + 4 * V, hh[1]);
                res_st<V>(hs + 5 * V, hh[2]);
            }
        }
    }

    /* wall row: rho_W from the wall-bound populations as updated (before they were rounded
     * to storage), then the gas-bound ones f = rho_W S(u_W) */
    __device__ __noinline__ void wall_fill(int s, const ResRow &rr, int rowi, int x0, int phase, const ResLat<R> &L)
    {
        const int w = (rr.flags & 2) ? 1 : 0, Q = h.q[s], nh = h.nh[s];
        const R nsgn = w == 0 ? R(1) : R(-1), rho0 = L.rho0;
        const Pop *tp = pops + s * LB_QMAX;
        const int off = rr.own * pitch + xoff + x0;
        const int ab = w == 0 ? 0 : Q - nh, ag = w == 0 ? Q - nh : 0;   /* wall-bound, gas-bound halves */
        const R *wb = reinterpret_cast<const R *>(sm + h.off_wall) + ((size_t)rr.wallord * h.nhmax * upr + x0 / V) * V;
        R num[V];
#pragma unroll
        for (int k = 0; k < V; ++k) num[k] = R(0);
#pragma unroll 6
        for (int i = 0; i < nh; ++i) {
            const Pop &p = tp[ab + i];
            const R xn = PO::cy(p) * nsgn;
            R d[V];
            if constexpr (EXACT) {
                T raw[V];
                res_ld<V>(plane(s, phys(s, ab + i, phase)) + off, raw);
#pragma unroll
                for (int k = 0; k < V; ++k) d[k] = dec(raw[k], PO::winv(p), rho0);
            } else {
                res_ld<V>(wb + (size_t)i * upr * V, d);
            }
#pragma unroll
            for (int k = 0; k < V; ++k) num[k] = fma(-xn * PO::w(p), d[k], num[k]);
        }
        const R uwx = L.uw_x[w], uwy = L.uw_y[w];
        const R usw = uwx * uwx + uwy * uwy;
        const R kd = L.kdiff[s][w], kout = L.kout[s][w];
        R rwd[V];
#pragma unroll
        for (int k = 0; k < V; ++k) rwd[k] = fma(rho0, kd, num[k]) / kout;   /* rho_W - rho0 */
        const uint16_t *to = pushes(rowi, 0);
#pragma unroll 2
        for (int i = 0; i < nh; ++i) {
            const int a = ag + i;
            const Pop &p = tp[a];
            const R ew = PO::cx(p) * uwx + PO::cy(p) * uwy;
            const R sm1 = ew + R(0.5) * (ew * ew - usw);    /* S / w - 1 */
            T e[V];
#pragma unroll
            for (int k = 0; k < V; ++k) e[k] = encode<ST>(fma(rwd[k] + rho0, sm1, rwd[k]), PO::w(p), rho0);
            const int ph = phys(s, a, phase);
            put(plane(s, ph), rr.own, x0, e);
            if (CL && (rr.flags & RES_PUSH)) push(s, ph, to, x0, e);
        }
    }

    /* ---- 2. views of shadow rows in the other set, one (unit, population) per thread ---- */
    __device__ void views(const int (&phase)[2])
    {
        const uint16_t *list = reinterpret_cast<const uint16_t *>(sm + h.off_shlist);
        const int q1 = h.q[1], q0 = h.q[0];
        const int n1 = h.nsh[1] * upr, n0 = h.nsh[0] * upr;   /* shadow units per own set */
        const int total = n0 * q1 + n1 * q0;
        for (int i = threadIdx.x; i < total; i += RES_THREADS) {
            const int s = i < n0 * q1 ? 0 : 1;   /* the rows' own set */
            const int t = 1 - s, k0 = s == 0 ? i : i - n0 * q1, n = s == 0 ? n0 : n1;
            const int b = k0 / n, un = k0 - b * n;
            const int ord = (s == 0 ? 0 : h.nsh[0]) + un / upr, x0 = (un % upr) * V;
            const int rowi = list[ord];
            const ResRow rr = rows[rowi];
            const R rho0 = lats[rr.lat].rho0;
            const R *hs = reinterpret_cast<const R *>(sm + h.off_herm) + ((size_t)ord * upr + x0 / V) * 6 * V;
            R c[6][V];
#pragma unroll
            for (int m = 0; m < 6; ++m) res_ld<V>(hs + m * V, c[m]);
            const Pop &p = pops[t * LB_QMAX + b];
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
            const int ph = phys(t, b, phase[t]);
            if (rr.view != RES_NONE) put(plane(t, ph), rr.view, x0, e);
            if (CL && (rr.flags & RES_PUSH)) push(t, ph, pushes(rowi, 1), x0, e);
        }
    }

    /* ---- 3. one round of the update: populations [a0, a1) of set s for 32 units ---- */
    __device__ __forceinline__ void update(int s, int chunk, int a0, int a1, int phase, uint32_t step_key, bool sr)
    {
        const int e = chunk * 32 + lane;
        if (e >= h.nunit[s]) return;
        int r, x0;
        locate(e, r, x0);
        const int rowi = (s ? h.nrow[0] : 0) + r;
        const ResRow rr = rows[rowi];
        const ResLat<R> &L = lats[rr.lat];
        const Pop *tp = pops + s * LB_QMAX;
        const R rho0 = L.rho0;
        const int n = V * h.nunit[s];
        R stt[5][V];
        {
            const R *st = state(s) + V * e;
#pragma unroll
            for (int i = 0; i < 5; ++i) res_ld<V>(st + i * n, stt[i]);
        }
        const int xb = xoff + x0;
        const int oo = rr.own * pitch + xb;
        const int om2 = rr.m2 * pitch + xb, om1 = rr.m1 * pitch + xb, op1 = rr.p1 * pitch + xb, op2 = rr.p2 * pitch + xb;
        /* x neighbours: the row's other end where the width is a whole number of units, the
         * images beside the row else */
        int ox[4];
        if constexpr (PAIR) {
            ox[0] = oo + ((xoff == 0 && x0 == 0) ? W - 2 : -2);
            ox[1] = oo + ((xoff == 0 && x0 + 4 == W) ? 4 - W : 4);
            ox[2] = ox[3] = 0;
        } else {
            const int ro = oo - x0;
            ox[0] = ro + (x0 >= 2 ? x0 - 2 : x0 - 2 + W);
            ox[1] = ro + (x0 >= 1 ? x0 - 1 : x0 - 1 + W);
            ox[2] = ro + (x0 + 1 < W ? x0 + 1 : x0 + 1 - W);
            ox[3] = ro + (x0 + 2 < W ? x0 + 2 : x0 + 2 - W);
        }
        const int wall = rr.flags & 3;
        const R wsgn = wall == 1 ? R(1) : (wall == 2 ? R(-1) : R(0));
        const int M = h.q[s] + h.K[s];
        int ph = phys(s, a0, phase);
        int pn = ph - h.K[s];
        if (pn < 0) pn += M;
        const uint32_t pstride = (uint32_t)h.nslot[s] * rowb;
        if constexpr (PAIR) {
            PairNode nd;
#pragma unroll
            for (int hh = 0; hh < 2; ++hh) {
                const int k = 2 * hh;
                nd.ux[hh] = make_float2(stt[0][k], stt[0][k + 1]);
                nd.uy[hh] = make_float2(stt[1][k], stt[1][k + 1]);
                nd.nom[hh] = make_float2(-stt[2][k], -stt[2][k + 1]);
                nd.P[hh] = make_float2(stt[2][k] * stt[3][k], stt[2][k + 1] * stt[3][k + 1]);
                nd.B[hh] = make_float2(stt[4][k], stt[4][k + 1]);
                if constexpr (FORCE) nd.dr[hh] = make_float2(L.dt * stt[3][k], L.dt * stt[3][k + 1]);
            }
            const float2 nrho02 = f2(-rho0);
            auto dec2 = [&](float2 raw, float2 winv2) -> float2 {
                if constexpr (ST == 1) return fma2(raw, winv2, nrho02);
                else return raw;
            };
#pragma unroll 1
            for (int a = a0; a < a1; ++a) {
                const RingPop &rp = tp[a];
                const T *pl = reinterpret_cast<const T *>(sm + h.off_plane[s] + (uint32_t)ph * pstride);
                T own[4], yv[3][4], hl[2], hr[2];
                const float cy = rp.cy2.x, cx = rp.cx2.x;
                ldn<4>(pl + oo, own);
                if (cy > 0.0f) {
                    ldn<4>(pl + om2, yv[0]);
                    ldn<4>(pl + om1, yv[1]);
                    ldn<4>(pl + op1, yv[2]);
                } else if (cy < 0.0f) {
                    ldn<4>(pl + op2, yv[0]);
                    ldn<4>(pl + op1, yv[1]);
                    ldn<4>(pl + om1, yv[2]);
                }
                if (cx != 0.0f) {
                    ld2(pl + ox[0], hl);
                    ld2(pl + ox[1], hr);
                }
                float2 v[2], c[2];
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) v[hh] = dec2(make_float2(to_r(own[2 * hh]), to_r(own[2 * hh + 1])), rp.winv2);
                PairC pc;
                PairC2 pc2;
                pc.cx2 = rp.cx2;
                pc.cy2 = rp.cy2;
                pc.ncx2 = rp.ncx2;
                pc.nacy2 = rp.nacy2;
                pc.ky2 = rp.ky2;
                pc.crx = -rp.ncx2.x;
                pc.kx = rp.kx;
                pc.ystep = cy != 0.0f;
                if constexpr (FORCE) pc2.gxi2 = f2(xi_dot(cx, cy, L.gx, L.gy));
                auto xh = [&](int i) -> float { return dec(i < 2 ? hl[i] : hr[i - 2], rp.winv2.x, rho0); };
                auto yw = [&](int hh, int i) -> float2 {
                    return dec2(make_float2(to_r(yv[i][2 * hh]), to_r(yv[i][2 * hh + 1])), rp.winv2);
                };
                pair_increment<FORCE>(pc, pc2, nd, v, xh, yw, c);
                float2 dn[2];
#pragma unroll
                for (int hh = 0; hh < 2; ++hh) dn[hh] = add2(v[hh], c[hh]);
                T ev[4];
                if constexpr (ST == 1) {
                    const float2 e0 = mul2(rp.w2, add2(f2(rho0), dn[0])), e1 = mul2(rp.w2, add2(f2(rho0), dn[1]));
                    ev[0] = e0.x, ev[1] = e0.y, ev[2] = e1.x, ev[3] = e1.y;
                } else {
                    ev[0] = from_r<T>(dn[0].x), ev[1] = from_r<T>(dn[0].y), ev[2] = from_r<T>(dn[1].x), ev[3] = from_r<T>(dn[1].y);
                }
                put(plane(s, pn), rr.own, x0, ev);
                if (rr.flags & (3 | RES_PUSH)) finish(s, a, pn, rr, rowi, x0, wsgn * cy, {dn[0].x, dn[0].y, dn[1].x, dn[1].y}, ev);
                ph = ph + 1 == M ? 0 : ph + 1;
                pn = pn + 1 == M ? 0 : pn + 1;
            }
        } else {
            const R ux = stt[0][0], uy = stt[1][0], om = stt[2][0], rho = stt[3][0], rhod = stt[4][0];
            const R usq = usq_of(ux, uy), gu = xi_dot(L.gx, L.gy, ux, uy);
#pragma unroll 2
            for (int a = a0; a < a1; ++a) {
                const Pop &p = tp[a];
                const T *pl = reinterpret_cast<const T *>(sm + h.off_plane[s] + (uint32_t)ph * pstride);
                const R winv = p.winv, crx = p.crx, cry = p.cry;
                const R v = dec(pl[oo], winv, rho0);
                R Dx = R(0), Dy = R(0);
                if (crx != R(0)) {
                    const R l[2] = {dec(pl[ox[0]], winv, rho0), dec(pl[ox[1]], winv, rho0)};
                    const R rr2[2] = {dec(pl[ox[2]], winv, rho0), dec(pl[ox[3]], winv, rho0)};
                    const R vv[1] = {v};
                    R D[1];
                    x_flux_diff<1>(crx, p.kx, l, vv, rr2, D);
                    Dx = D[0];
                }
                if (cry > R(0)) {
                    const R ym2 = dec(pl[om2], winv, rho0), ym1 = dec(pl[om1], winv, rho0), yp1 = dec(pl[op1], winv, rho0);
                    const R d0 = ym1 - ym2, d1 = v - ym1, d2 = yp1 - v, n1 = neg_part(d1);
                    Dy = fma(p.ky, minmod_n(d1, d2, n1, neg_part(d2)) - minmod_n(d0, d1, neg_part(d0), n1), d1);
                } else if (cry < R(0)) {
                    const R ym1 = dec(pl[om1], winv, rho0), yp1 = dec(pl[op1], winv, rho0), yp2 = dec(pl[op2], winv, rho0);
                    const R e0 = v - ym1, e1 = yp1 - v, e2 = yp2 - yp1, n1 = neg_part(e1);
                    Dy = fma(-p.ky, minmod_n(e1, e2, n1, neg_part(e2)) - minmod_n(e0, e1, neg_part(e0), n1), e1);
                }
                const R eu = xi_dot(p.cx, p.cy, ux, uy);
                R inc = om * (deq(rhod, rho, eu, usq) - v);
                inc = fma(-crx, Dx, inc);
                inc = fma(-cry, Dy, inc);
                if constexpr (FORCE) inc = force_inc(L.dt * rho, xi_dot(p.cx, p.cy, L.gx, L.gy), eu, gu, inc);
                const R dn = v + inc;
                T ev[1];
                if (sr) ev[0] = encode_sr<ST>(dn, p.w, rho0, sr_bits(x0, (int)rr.j, W, a, step_key));
                else ev[0] = encode<ST>(dn, p.w, rho0);
                put(plane(s, pn), rr.own, x0, ev);
                if (rr.flags & (3 | RES_PUSH)) finish(s, a, pn, rr, rowi, x0, wsgn * p.cy, {dn}, ev);
                ph = ph + 1 == M ? 0 : ph + 1;
                pn = pn + 1 == M ? 0 : pn + 1;
            }
        }
    }
    /* wall rows keep the unrounded wall-bound values; rows next to another block's are
     * stored there too */
    __device__ __forceinline__ void finish(int s, int a, int pn, const ResRow &rr, int rowi, int x0, R xn, const R (&dn)[V],
                                           const T (&ev)[V])
    {
        if (!EXACT && xn < R(0)) {
            const int i = (rr.flags & 2) ? a - (h.q[s] - h.nh[s]) : a;
            R *wb = reinterpret_cast<R *>(sm + h.off_wall) + (((size_t)rr.wallord * h.nhmax + i) * upr + x0 / V) * V;
            res_st<V>(wb, dn);
        }
        if (CL && (rr.flags & RES_PUSH)) push(s, pn, pushes(rowi, 0), x0, ev);
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
    extern __shared__ __align__(16) unsigned char res_smem[];
    ResHead &h = *reinterpret_cast<ResHead *>(res_smem);
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
        RT rt(h, res_smem);
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
            const uint4 *src = reinterpret_cast<const uint4 *>(&tabs[ids[0]]);
            for (int k = tid; k < (int)(sizeof(RingTab) / 16); k += RES_THREADS) reinterpret_cast<uint4 *>(pops)[k] = src[k];
        } else {
            const StepParams<R> &p = par2[2 * (size_t)ids[0] + base];
            for (int k = tid; k < 2 * LB_QMAX; k += RES_THREADS) {
                const SetConst<R> &c = p.set[k / LB_QMAX];
                const int a = k % LB_QMAX;
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
                T *row = rt.plane(s, a) + rt.rows[r0 + r].own * rt.pitch + rt.xoff;
                row[x] = v;
                if (rt.xoff != 0) {
                    if (x < 2) row[x + W] = v;
                    if (x >= W - 2) row[x - W] = v;
                }
                if constexpr (CL) {
                    if (rt.rows[r0 + r].flags & RES_PUSH) {
                        const uint16_t *to = rt.pushes(r0 + r, 0);
                        for (int t = 0; t < 2; ++t) {
                            const int rk = to[2 * t];
                            if (rk == RES_NONE) continue;
                            const ResRank &kk = h.rank[rk];
                            T *local = reinterpret_cast<T *>(res_smem + kk.off_plane[s] + (uint32_t)a * kk.nslot[s] * rt.rowb);
                            T *rrow = cg::this_cluster().map_shared_rank(local, rk) + to[2 * t + 1] * rt.pitch + rt.xoff;
                            rrow[x] = v;
                            if (rt.xoff != 0) {
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
        for (int st = 0;; ++st) {
            if (st == 0) rt.template moments<false>(phase);
            else rt.template moments<true>(phase);
            __syncthreads();
            if (st == nsteps) break;
            rt.views(phase);
            if constexpr (CL) cg::this_cluster().sync();
            else __syncthreads();
            for (int rd = 0; rd < h.rounds; ++rd) {
                const int nc1 = (h.nunit[1] + 31) / 32, nc0 = (h.nunit[0] + 31) / 32;
                const int u1 = nc1 * h.G[1], u0 = nc0 * h.G[0];
                for (int u = rt.warp; u < u1 + u0; u += RES_WARPS) {
                    const int s = u < u1 ? 1 : 0;
                    const int k = s ? u : u - u1, nc = s ? nc1 : nc0;
                    const int g = k / nc, chunk = k - g * nc;
                    const int lo = rd * h.K[s], hi = min(h.q[s], lo + h.K[s]);
                    const int per = (h.K[s] + h.G[s] - 1) / h.G[s];
                    const int a0 = lo + g * per, a1 = min(hi, a0 + per);
                    if (a0 < a1) rt.update(s, chunk, a0, a1, phase[s], step0 + (uint32_t)st + 1u, sr);
                }
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
                        const ResRow rr = rt.rows[r0 + r];
                        if (view && !(rr.flags & RES_SHADOW)) continue;
                        const ResGRow g = grow[r0 + r];
                        const StepParams<R> &p = par2[2 * (size_t)g.lat + sel];
                        T v;
                        if (!view) {
                            v = rt.plane(t, rt.phys(t, a, phase[t]))[rr.own * rt.pitch + rt.xoff + x];
                        } else {   /* as views() formed it */
                            const R *hs = reinterpret_cast<const R *>(res_smem + h.off_herm) +
                                          ((size_t)rr.shord * rt.upr + x / RT::V) * 6 * RT::V + x % RT::V;
                            const typename RT::Pop &pc = pops[t * LB_QMAX + a];
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
                    const int off = rt.rows[r0 + r].own * rt.pitch + rt.xoff + x;
                    for (int a = 0; a < q; ++a) {
                        const typename RT::Pop &pc = pops[s * LB_QMAX + a];
                        using PO = typename RT::PO;
                        const R d = decode<ST>(rt.plane(s, rt.phys(s, a, phase[s]))[off], PO::winv(pc), rho0);
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
    /* raised on every launch: the limit is per function and device, and the call is cheap
     * next to a launch of many steps */
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)a.plan->smem) != cudaSuccess) {
        cudaGetLastError();
        return -1;
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
        if (a.plan->cluster > 8 &&
            cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
            cudaGetLastError();
            return -1;
        }
    } else {
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
