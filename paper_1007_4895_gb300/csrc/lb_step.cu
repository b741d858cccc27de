/*
 * lb_step.cu -- the small passes that complete a time level (interface rows of mode A,
 * pressure columns, rebuilt interface views after the state is replaced) and the
 * dispatch of the step kernel (lb_step_impl.cuh) to its per-storage instantiations.
 */
#include <cuda_runtime.h>

#include <type_traits>

#include "lb_common.cuh"
#include "lb_pressure.cuh"
#include "lb_tma.h"

namespace lbk {

template <int ST>
void launch_step_store(const StepParams<typename Store<ST>::R> &p, void *stream);
template <int ST>
void launch_step_desc_store(const StepParams<typename Store<ST>::R> &p, int n, void *stream);
template <int ST>
void launch_step_split_store(const StepParams<typename Store<ST>::R> &p, int rb, const int2 *edge, int n_edge,
                             void *stream, void *edge_stream);
template <int ST>
void launch_pair_store(const StepParams<float> &p, void *stream);
template <int ST>
void launch_ring_store(const StepParams<float> &p, void *stream);
template <int ST, int Q1>
void launch_ring_units_store(const StepParams<float> &p, const RingTab &tab, const RowQueues &rq, int nblocks,
                             void *stream);
template <int ST, int Q1>
int launch_tiles_store(const StepParams<float> &p, const RingTab &tab, const TileMaps &maps, const int4 *units, int nunits,
                       int n1, uint32_t *ctr, int *err, void *stream);
template <int ST, int Q1>
int launch_ring_batch_store(const StepParams<float> *params, const RingTab *tabs, const uint32_t *items,
                            const int2 *ranges, const int *order, int n, int nsteps, int base, int advance,
                            unsigned int *queue, bool force, int grid, int *grid_out, void *stream);

/* ---------------------------------------------------------------- mode A -- */

/* Sec. 2.2: interface row I gets, in each set s, f_eq^s(rho_I, u_I) + f_neq^s of the
 * neighbour on s's own side, with rho_I, u_I the means of its two neighbours; the node
 * one beyond I on the other side gets a copy (what a reader reaching past I sees). */
template <int ST>
__global__ void iface_kernel(const __grid_constant__ StepParams<typename Store<ST>::R> p)
{
    using T = typename Store<ST>::T;
    using R = typename Store<ST>::R;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= p.nx || blockIdx.y >= (unsigned)p.n_iface) return;
    const int I = p.iface_row[blockIdx.y];
    const uint8_t flags = p.tmap[(size_t)I * p.ntx + x / LB_TILE_X];
    const int jh = (flags & LB_TILE_NEAR_H) ? I - 1 : I + 1;
    const int jl = (flags & LB_TILE_NEAR_H) ? I + 1 : I - 1;
    const size_t plane = p.plane;
    const R rho0 = p.rho0;
    R rhod[2], u[2][2];
    const int rows[2] = {jl, jh};
    for (int s = 0; s < 2; ++s) {
        const SetConst<R> &c = p.set[s];
        const T *f = static_cast<const T *>(p.fout[s]) + (size_t)rows[s] * p.pitch + x + LB_GHOST;
        R r = R(0), mx = R(0), my = R(0);
        for (int a = 0; a < c.q; ++a) {
            R d = dec_at<ST>(p, f[a * plane], c.winv[a], x + LB_GHOST);
            r = fma(c.w[a], d, r);
            mx = fma(c.wcx[a], d, mx);
            my = fma(c.wcy[a], d, my);
        }
        rhod[s] = r;
        u[s][0] = mx / (rho0 + r);
        u[s][1] = my / (rho0 + r);
    }
    const R rIdev = R(0.5) * (rhod[0] + rhod[1]);
    const R rI = rho0 + rIdev;
    const R uIx = R(0.5) * (u[0][0] + u[1][0]), uIy = R(0.5) * (u[0][1] + u[1][1]);
    const R usI = uIx * uIx + uIy * uIy;
    for (int s = 0; s < 2; ++s) {
        const SetConst<R> &c = p.set[s];
        const T *fn = static_cast<const T *>(p.fout[s]) + (size_t)rows[s] * p.pitch + x + LB_GHOST;
        T *fo = static_cast<T *>(p.fout[s]);
        const int beyond = rows[1 - s];
        const R rn = rho0 + rhod[s], usn = u[s][0] * u[s][0] + u[s][1] * u[s][1];
        for (int a = 0; a < c.q; ++a) {
            const R dnb = dec_at<ST>(p, fn[a * plane], c.winv[a], x + LB_GHOST);
            const R eI = c.cx[a] * uIx + c.cy[a] * uIy;
            const R en = c.cx[a] * u[s][0] + c.cy[a] * u[s][1];
            const R d = deq(rIdev, rI, eI, usI) + (dnb - deq(rhod[s], rn, en, usn));
            const T e = enc_at<ST>(p, d, c.w[a], x + LB_GHOST);
            put1r(p, fo + a * plane + (size_t)I * p.pitch, x, I, e);
            put1r(p, fo + a * plane + (size_t)beyond * p.pitch, x, beyond, e);
        }
    }
}

/* ------------------------------------------------------- pressure columns -- */

/* One warp per (row, side) of the pressure columns (lb_pressure.cuh). */
template <int ST>
__global__ void pressure_kernel(const __grid_constant__ StepParams<typename Store<ST>::R> p)
{
    const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int side = blockIdx.y;
    if (j >= p.ny || !p.pressure[side]) return;   /* uniform over the warp */
    pressure_row<ST>(p, j, side);
}

/* ------------------------------------------------ interface views, ghosts -- */

/* Rebuild every node of a mode-B shadow tile in the other set from its current state
 * (used after the state or the map is replaced, not inside a step). */
template <int ST>
__global__ void shadows_kernel(const __grid_constant__ StepParams<typename Store<ST>::R> p)
{
    using T = typename Store<ST>::T;
    using R = typename Store<ST>::R;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y;
    if (x >= p.nx) return;
    const uint8_t flags = p.tmap[(size_t)j * p.ntx + x / LB_TILE_X];
    if (!(flags & LB_TILE_SHADOW)) return;
    const int s = flags & LB_TILE_HIGH;
    const SetConst<R> &c = p.set[s];
    const SetConst<R> &ct = p.set[1 - s];
    const size_t plane = p.plane;
    const T *f = static_cast<const T *>(p.fout[s]) + (size_t)j * p.pitch + x + LB_GHOST;
    R h[6] = {R(0), R(0), R(0), R(0), R(0), R(0)};
    for (int a = 0; a < c.q; ++a) hermite_acc(c, a, dec_at<ST>(p, f[a * plane], c.winv[a], x + LB_GHOST), h);
    T *ft = static_cast<T *>(p.fout[1 - s]);
    for (int b = 0; b < ct.q; ++b)
        put1r(p, ft + b * plane + (size_t)j * p.pitch, x, j, enc_at<ST>(p, hermite_rebuild(ct, b, h), ct.w[b], x + LB_GHOST));
}

/* ----------------------------------------------- D2Q9 stream and collide -- */

/* The D2Q9 reduction of the Sec. 3.1 update at Courant number one (dt = h / sqrt(3),
 * abscissae +-sqrt(3)): every population moves exactly one node along sign(xi) per step
 * (stream), then relaxes towards Eq. (demoeq) with the Eq. (demoforce) force at the
 * streamed state (collide). Periodic lattice of one set. The ghost rows and columns hold
 * the periodic images, so the pull needs no index logic.
 *
 * Odd steps walk the rows from the top: the rows a step wrote last are still in L2 (129
 * MB) when the next step reads them first, which saves DRAM traffic once the two levels do
 * not fit (the kernel of two nodes per thread; in FP64, bound by its units, it gained nothing:
 * 2048 x 1024 758.4 and 757.7 us). */
template <typename R>
__device__ __forceinline__ int stream_row(const StepParams<R> &p)
{
    return (p.step_key & 1u) ? p.ny - 1 - (int)blockIdx.y : (int)blockIdx.y;
}

/* One thread per node: FP64, and boxes of STREAM_ONE nodes at most. */
template <int ST>
__global__ void __launch_bounds__(128) exact_stream_kernel(const __grid_constant__ StepParams<typename Store<ST>::R> p)
{
    using T = typename Store<ST>::T;
    using R = typename Store<ST>::R;
    const int x = blockIdx.x * blockDim.x + threadIdx.x, j = blockIdx.y;
    if (x >= p.nx) return;
    /* the population loops are unrolled, so the set's constants are read from the
     * parameter block at fixed offsets; population a = 3 iy + ix over ascending
     * abscissae moves by (ix - 1, iy - 1) */
    const SetConst<R> &c = p.set[0];
    const T *fin = static_cast<const T *>(p.fin[0]);
    T *fout = static_cast<T *>(p.fout[0]);
    const size_t plane = p.plane;
    const R rho0 = p.rho0;
    R d[9], rd = R(0), jx = R(0), jy = R(0);
#pragma unroll
    for (int a = 0; a < 9; ++a) {
        const int sx = a % 3 - 1, sy = a / 3 - 1;
        const int col = x - sx + LB_GHOST;
        d[a] = dec_at<ST>(p, fin[a * plane + (ptrdiff_t)(j - sy) * p.pitch + col], c.winv[a], col);
        rd = fma(c.w[a], d[a], rd);
        jx = fma(c.wcx[a], d[a], jx);
        jy = fma(c.wcy[a], d[a], jy);
    }
    const R rho = rho0 + rd, inv = R(1) / rho;
    const R ux = jx * inv, uy = jy * inv;
    const R usq = usq_of(ux, uy), om = p.dt / tau_of(p, inv), gu = xi_dot(p.gx, p.gy, ux, uy);
    int img[2];
    /* a node whose value has no ghost copy: stored once */
    const bool plain = row_images(p, j, img) == 0 && x >= LB_GHOST && x < p.nx - LB_GHOST;
    T *row = fout + (size_t)j * p.pitch;
#pragma unroll
    for (int a = 0; a < 9; ++a) {
        const R eu = xi_dot(c.cx[a], c.cy[a], ux, uy);
        R inc = om * (deq(rd, rho, eu, usq) - d[a]);
        if (p.has_force) inc = force_inc(p.dt * rho, xi_dot(c.cx[a], c.cy[a], p.gx, p.gy), eu, gu, inc);
        const T e = enc_at<ST>(p, d[a] + inc, c.w[a], x + LB_GHOST);
        if (plain) row[a * plane + x + LB_GHOST] = e;
        else put1r(p, row + a * plane, x, j, e);
    }
}

/* FP32 and 16-bit storage, larger boxes: two neighbouring nodes per thread in packed two-wide FP32
 * arithmetic, the same operations per node as above (the terms whose abscissa is zero
 * left out: they add exact zeros), so the same values. One node per thread was bound by
 * instruction issue (480 a node, 84 % of the issue slots: 64-bit addresses and scalar
 * arithmetic), not by memory. Per-column reference density: COL. 2048 x 1024, FP32
 * deviations, 20 steps and the fields: 788 -> 583 us. */
template <int ST, bool COL>
__global__ void __launch_bounds__(128) exact_stream_pair_kernel(const __grid_constant__ StepParams<float> p)
{
    using T = typename Store<ST>::T;
    const int x = 2 * (blockIdx.x * 128 + threadIdx.x), j = stream_row(p);
    if (x >= p.nx) return;
    const SetConst<float> &c = p.set[0];
    const T *__restrict__ fin = static_cast<const T *>(p.fin[0]) + (ptrdiff_t)j * p.pitch + x + LB_GHOST;
    const ptrdiff_t plane = (ptrdiff_t)p.plane;
    const float rho0 = p.rho0;
    auto f2 = [](float v) { return make_float2(v, v); };
    float dl[4] = {0.0f, 0.0f, 0.0f, 0.0f};   /* delta at columns x - 1 .. x + 2 */
    if constexpr (COL) {
#pragma unroll
        for (int i = 0; i < 4; ++i) dl[i] = p.dcol[x + LB_GHOST - 1 + i];
    }
    T raw[9][2];
#pragma unroll
    for (int a = 0; a < 9; ++a) {
        const int sx = a % 3 - 1, sy = a / 3 - 1;
        const T *q = fin + a * plane - sy * (ptrdiff_t)p.pitch - sx;
        if (sx == 0) {
            ld2(q, raw[a]);
        } else {
            raw[a][0] = q[0];
            raw[a][1] = q[1];
        }
    }
    float2 d[9], rd = f2(0.0f), jx = f2(0.0f), jy = f2(0.0f);
#pragma unroll
    for (int a = 0; a < 9; ++a) {
        const int sx = a % 3 - 1, sy = a / 3 - 1;
        const float2 r = make_float2(to_r(raw[a][0]), to_r(raw[a][1]));
        if constexpr (ST == 1) d[a] = __ffma2_rn(r, f2(c.winv[a]), f2(-rho0));
        else if constexpr (COL) d[a] = __fadd2_rn(r, make_float2(dl[1 - sx], dl[2 - sx]));
        else d[a] = r;
        rd = __ffma2_rn(f2(c.w[a]), d[a], rd);
        if (sx != 0) jx = __ffma2_rn(f2(c.wcx[a]), d[a], jx);
        if (sy != 0) jy = __ffma2_rn(f2(c.wcy[a]), d[a], jy);
    }
    const float2 rho = __fadd2_rn(f2(rho0), rd);
    const float2 inv = make_float2(1.0f / rho.x, 1.0f / rho.y);
    const float2 ux = __fmul2_rn(jx, inv), uy = __fmul2_rn(jy, inv);
    const float2 usq = __ffma2_rn(uy, uy, __fmul2_rn(ux, ux));
    const float2 nusq = make_float2(-usq.x, -usq.y);
    const float2 om = make_float2(p.dt / tau_of(p, inv.x), p.dt / tau_of(p, inv.y));
    float2 gu = f2(0.0f), dtr = f2(0.0f);
    if (p.has_force) {
        gu = __ffma2_rn(f2(p.gy), uy, __fmul2_rn(f2(p.gx), ux));
        dtr = __fmul2_rn(f2(p.dt), rho);
    }
    int img[2];
    const bool plain = row_images(p, j, img) == 0 && x >= LB_GHOST && x + 1 < p.nx - LB_GHOST;
    T *row = static_cast<T *>(p.fout[0]) + (size_t)j * p.pitch;
#pragma unroll
    for (int a = 0; a < 9; ++a) {
        const int sx = a % 3 - 1, sy = a / 3 - 1;
        float2 eu = f2(0.0f);
        if (sx != 0 && sy != 0) eu = __ffma2_rn(f2(c.cy[a]), uy, __fmul2_rn(f2(c.cx[a]), ux));
        else if (sx != 0) eu = __fmul2_rn(f2(c.cx[a]), ux);
        else if (sy != 0) eu = __fmul2_rn(f2(c.cy[a]), uy);
        const float2 de = __ffma2_rn(rho, __ffma2_rn(f2(0.5f), __ffma2_rn(eu, eu, nusq), eu), rd);
        /* scalar multiplies: a packed multiply would be fused with the packed add below */
        const float2 df = __fadd2_rn(de, make_float2(-d[a].x, -d[a].y));
        float2 inc = make_float2(__fmul_rn(om.x, df.x), __fmul_rn(om.y, df.y));
        if (p.has_force) {
            const float2 gxi = f2(xi_dot(c.cx[a], c.cy[a], p.gx, p.gy));
            inc = __ffma2_rn(dtr, __fadd2_rn(__ffma2_rn(gxi, eu, gxi), make_float2(-gu.x, -gu.y)), inc);
        }
        float2 v = __fadd2_rn(d[a], inc);
        if constexpr (COL) v = __fadd2_rn(v, make_float2(-dl[1], -dl[2]));
        if constexpr (ST == 1) v = __fmul2_rn(f2(c.w[a]), __fadd2_rn(f2(rho0), v));
        const T e[2] = {from_r<T>(v.x), from_r<T>(v.y)};
        T *q = row + a * plane;
        if (plain) {
            st2(q + x + LB_GHOST, e);
        } else {
            put1r(p, q, x, j, e[0]);
            if (x + 1 < p.nx) put1r(p, q, x + 1, j, e[1]);
        }
    }
}

/* ------------------------------------------------------ carried moments -- */

/* A quad's moments in population order, node_moments() per node: twelve planes' vectors are
 * on their way at a time. */
template <int ST, int Q>
__device__ __forceinline__ void quad_moments(const typename Store<ST>::T *f, size_t plane,
                                             const MomC<typename Store<ST>::R> *mc, typename Store<ST>::R rho0, bool col,
                                             const typename Store<ST>::R delta[4], typename Store<ST>::R rd[4],
                                             typename Store<ST>::R jx[4], typename Store<ST>::R jy[4])
{
    using T = typename Store<ST>::T;
    using R = typename Store<ST>::R;
    constexpr int C = Q == 36 ? 12 : Q == 16 ? 8 : 9;
#pragma unroll
    for (int i = 0; i < 4; ++i) rd[i] = jx[i] = jy[i] = R(0);
#pragma unroll 1
    for (int a0 = 0; a0 < Q; a0 += C) {
        T v[C][4];
#pragma unroll
        for (int k = 0; k < C; ++k) ld4(f + (a0 + k) * plane, v[k]);
#pragma unroll
        for (int k = 0; k < C; ++k) {
            const MomC<R> m = mc[a0 + k];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const R d = col ? decode_col<ST>(v[k][i], m.winv, rho0, delta[i]) : decode<ST>(v[k][i], m.winv, rho0);
                rd[i] = fma(m.w, d, rd[i]);
                jx[i] = fma(m.wcx, d, jx[i]);
                jy[i] = fma(m.wcy, d, jy[i]);
            }
        }
    }
}

/* Carried moments of the written level, sum w d, sum w xi_x d, sum w xi_y d per node
 * from its stored populations in population order. Runs once per uploaded or initialised
 * state, before the first step. Bound by memory latency: one node per thread had a chain of
 * 36 four-byte loads; a quad per thread loads 16 bytes a plane (a quad lies in one tile, so
 * in one set, and starts at a multiple of 16 bytes).
 * Upload of the 16384 x 128 channel's state (FP32 deviations, 122 MB): 720 us before, 651
 * with quads, of which the copy from the host takes about 600. */
template <int ST>
__global__ void __launch_bounds__(128) aux_kernel(const __grid_constant__ StepParams<typename Store<ST>::R> p)
{
    using T = typename Store<ST>::T;
    using R = typename Store<ST>::R;
    __shared__ PopC<R> pcs[2][LB_QMAX];
    __shared__ MomC<R> mcs[2][LB_QMAX];
    stage_consts(p, pcs, mcs, threadIdx.x, blockDim.x);
    __syncthreads();
    const unsigned nq = ((unsigned)p.nx + 3) / 4, k = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = (int)(k / nq), x = (int)(k - (unsigned)j * nq) * 4;
    if (j >= p.ny) return;
    const int s = p.tmap[(size_t)j * p.ntx + x / LB_TILE_X] & LB_TILE_HIGH;
    const T *f = static_cast<const T *>(p.fout[s]) + (size_t)j * p.pitch + x + LB_GHOST;
    R delta[4], rd[4], jx[4], jy[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) delta[i] = p.dcol && x + i < p.nx ? p.dcol[x + i + LB_GHOST] : R(0);
    const int q = p.set[s].q;
    if (q == 9) quad_moments<ST, 9>(f, p.plane, mcs[s], p.rho0, p.dcol != nullptr, delta, rd, jx, jy);
    else if (q == 16) quad_moments<ST, 16>(f, p.plane, mcs[s], p.rho0, p.dcol != nullptr, delta, rd, jx, jy);
    else quad_moments<ST, 36>(f, p.plane, mcs[s], p.rho0, p.dcol != nullptr, delta, rd, jx, jy);
    R *aout = static_cast<R *>(p.aux_out) + (size_t)j * p.pitch + x;
    const size_t ap = (size_t)p.pitch * p.ny;
    if (x + 3 < p.nx) {
        st4(aout, rd);
        st4(aout + ap, jx);
        st4(aout + 2 * ap, jy);
        return;
    }
    for (int i = 0; x + i < p.nx; ++i) {
        aout[i] = rd[i];
        aout[ap + i] = jx[i];
        aout[2 * ap + i] = jy[i];
    }
}

/* ------------------------------------------------------------- launchers -- */

template <typename R>
struct StoreFor;

#define LB_DISPATCH(store, ...)                                   \
    switch (store) {                                               \
        case 0: { constexpr int ST = 0; __VA_ARGS__; } break;             \
        case 1: { constexpr int ST = 1; __VA_ARGS__; } break;             \
        case 2: { constexpr int ST = 2; __VA_ARGS__; } break;             \
        case 3: { constexpr int ST = 3; __VA_ARGS__; } break;             \
        default: { constexpr int ST = 4; __VA_ARGS__; } break;            \
    }

template <typename R, int ST>
constexpr bool store_matches()
{
    return std::is_same<R, typename Store<ST>::R>::value;
}

template <typename R>
void launch_step(int store, const StepParams<R> &p, void *stream)
{
    LB_DISPATCH(store, if constexpr (store_matches<R, ST>()) launch_step_store<ST>(p, stream));
}

void launch_ring(int store, const StepParams<float> &p, void *stream)
{
    switch (store) {
        case 1: launch_ring_store<1>(p, stream); break;
        case 2: launch_ring_store<2>(p, stream); break;
        case 3: launch_ring_store<3>(p, stream); break;
        case 4: launch_ring_store<4>(p, stream); break;
        default: break;
    }
}

void launch_ring_units(int store, const StepParams<float> &p, const RingTab &tab, const RowQueues &rq, int nblocks,
                       void *stream)
{
    const bool q36 = p.set[1].q == 36;
    switch (store) {
        case 1: (q36 ? launch_ring_units_store<1, 36> : launch_ring_units_store<1, 16>)(p, tab, rq, nblocks, stream); break;
        case 2: (q36 ? launch_ring_units_store<2, 36> : launch_ring_units_store<2, 16>)(p, tab, rq, nblocks, stream); break;
        case 3: (q36 ? launch_ring_units_store<3, 36> : launch_ring_units_store<3, 16>)(p, tab, rq, nblocks, stream); break;
        case 4: (q36 ? launch_ring_units_store<4, 36> : launch_ring_units_store<4, 16>)(p, tab, rq, nblocks, stream); break;
        default: break;
    }
}

int launch_tiles(int store, const StepParams<float> &p, const RingTab &tab, const TileMaps &maps, const int4 *units,
                 int nunits, int n1, uint32_t *ctr, int *err, void *stream)
{
    const bool q36 = p.set[1].q == 36;
#define LB_TL(ST) (q36 ? launch_tiles_store<ST, 36> : launch_tiles_store<ST, 16>)(p, tab, maps, units, nunits, n1, ctr, err, stream)
    switch (store) {
        case 1: return LB_TL(1);
        case 2: return LB_TL(2);
        case 3: return LB_TL(3);
        case 4: return LB_TL(4);
        default: return -1;
    }
#undef LB_TL
}

int launch_ring_batch(int store, int q1, const StepParams<float> *params, const RingTab *tabs, const uint32_t *items,
                      const int2 *ranges, const int *order, int n, int nsteps, int base, int advance,
                      unsigned int *queue, bool force, int grid, int *grid_out, void *stream)
{
    const bool q36 = q1 == 36;
    if (!q36 && q1 != 16) return -1;
#define LB_RB(ST) (q36 ? launch_ring_batch_store<ST, 36> : launch_ring_batch_store<ST, 16>)( \
        params, tabs, items, ranges, order, n, nsteps, base, advance, queue, force, grid, grid_out, stream)
    switch (store) {
        case 1: return LB_RB(1);
        case 2: return LB_RB(2);
        case 3: return LB_RB(3);
        case 4: return LB_RB(4);
        default: return -1;
    }
#undef LB_RB
}

void launch_pair(int store, const StepParams<float> &p, void *stream)
{
    switch (store) {
        case 1: launch_pair_store<1>(p, stream); break;
        case 2: launch_pair_store<2>(p, stream); break;
        case 3: launch_pair_store<3>(p, stream); break;
        case 4: launch_pair_store<4>(p, stream); break;
        default: break;
    }
}

/* One node per thread up to here: a small box is bound by the chain of one thread, which two
 * nodes lengthen (us a step, FP32 deviations, two nodes / one: 64 x 16 6.2 / 4.2, 128 x 128 6.2 /
 * 5.0, 513 x 257 6.8 / 6.2, 512 x 512 8.2 / 8.3, 1024 x 512 10.3 / 12.4); the same bits. */
constexpr long long STREAM_ONE = 1 << 18;
template <typename R>
void launch_exact_stream(int store, const StepParams<R> &p, void *stream)
{
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const dim3 one((p.nx + 127) / 128, p.ny);
    if constexpr (std::is_same<R, double>::value) {
        exact_stream_kernel<0><<<one, 128, 0, st>>>(p);
    } else if ((long long)p.nx * p.ny <= STREAM_ONE) {
        LB_DISPATCH(store, if constexpr (store_matches<R, ST>()) exact_stream_kernel<ST><<<one, 128, 0, st>>>(p));
    } else {
        const dim3 grid((p.nx + 255) / 256, p.ny);
        LB_DISPATCH(store, if constexpr (store_matches<R, ST>()) {
            if constexpr (Store<ST>::dev) {
                if (p.dcol) {
                    exact_stream_pair_kernel<ST, true><<<grid, 128, 0, st>>>(p);
                    return;
                }
            }
            exact_stream_pair_kernel<ST, false><<<grid, 128, 0, st>>>(p);
        });
    }
}

template <typename R>
void launch_step_desc(int store, const StepParams<R> &p, int n, void *stream)
{
    LB_DISPATCH(store, if constexpr (store_matches<R, ST>()) launch_step_desc_store<ST>(p, n, stream));
}

template <int ST>
int launch_batch_store(const void *params, const int *order, int n, int nsteps, int base, int advance,
                       unsigned int *queue, int threads, int grid, void *stream);
template <int ST>
int batch_blocks_per_sm(int threads);

int launch_batch(int store, const void *params, const int *order, int n, int nsteps, int base, int advance,
                 unsigned int *queue, int threads, int grid, void *stream)
{
    int r = -1;
    LB_DISPATCH(store, r = launch_batch_store<ST>(params, order, n, nsteps, base, advance, queue, threads, grid, stream));
    return r;
}

int batch_blocks(int store, int threads)
{
    int r = 0;
    LB_DISPATCH(store, r = batch_blocks_per_sm<ST>(threads));
    return r;
}

template <typename R>
void launch_step_split(int store, const StepParams<R> &p, int rb, const int2 *edge, int n_edge, void *stream,
                       void *edge_stream)
{
    LB_DISPATCH(store, if constexpr (store_matches<R, ST>())
                           launch_step_split_store<ST>(p, rb, edge, n_edge, stream, edge_stream));
}

template <typename R>
void launch_iface(int store, const StepParams<R> &p, void *stream)
{
    if (p.n_iface <= 0) return;
    dim3 grid((p.nx + 127) / 128, p.n_iface);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    LB_DISPATCH(store, if constexpr (store_matches<R, ST>()) iface_kernel<ST><<<grid, 128, 0, st>>>(p));
}

template <typename R>
void launch_pressure(int store, const StepParams<R> &p, void *stream)
{
    if (!p.pressure[0] && !p.pressure[1]) return;
    dim3 grid((p.ny + 3) / 4, 2);   /* four warps (rows) per block */
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    LB_DISPATCH(store, if constexpr (store_matches<R, ST>()) pressure_kernel<ST><<<grid, 128, 0, st>>>(p));
}

template <typename R>
void launch_shadows(int store, const StepParams<R> &p, void *stream)
{
    dim3 grid((p.nx + 127) / 128, p.ny);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    LB_DISPATCH(store, if constexpr (store_matches<R, ST>()) shadows_kernel<ST><<<grid, 128, 0, st>>>(p));
}

template void launch_step<float>(int, const StepParams<float> &, void *);
template void launch_step<double>(int, const StepParams<double> &, void *);
template void launch_exact_stream<float>(int, const StepParams<float> &, void *);
template void launch_exact_stream<double>(int, const StepParams<double> &, void *);
template void launch_step_desc<float>(int, const StepParams<float> &, int, void *);
template void launch_step_desc<double>(int, const StepParams<double> &, int, void *);
template void launch_step_split<float>(int, const StepParams<float> &, int, const int2 *, int, void *, void *);
template void launch_step_split<double>(int, const StepParams<double> &, int, const int2 *, int, void *, void *);
template void launch_iface<float>(int, const StepParams<float> &, void *);
template void launch_iface<double>(int, const StepParams<double> &, void *);



template <typename R>
void launch_aux(int store, const StepParams<R> &p, void *stream)
{
    const long long items = (long long)((p.nx + 3) / 4) * p.ny;
    if (items <= 0) return;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    LB_DISPATCH(store, if constexpr (store_matches<R, ST>())
                           aux_kernel<ST><<<(unsigned)((items + 127) / 128), 128, 0, st>>>(p));
}

template void launch_aux<float>(int, const StepParams<float> &, void *);
template void launch_aux<double>(int, const StepParams<double> &, void *);
template void launch_pressure<float>(int, const StepParams<float> &, void *);
template void launch_pressure<double>(int, const StepParams<double> &, void *);
template void launch_shadows<float>(int, const StepParams<float> &, void *);
template void launch_shadows<double>(int, const StepParams<double> &, void *);

}  // namespace lbk
