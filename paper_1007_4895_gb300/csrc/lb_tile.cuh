/*
 * lb_tile.cuh -- layout 10 on tiles fed by the tensor memory accelerator.
 *
 * The row kernel of lb_ring2.cuh is bound by memory latency and by what its per-thread
 * ring of copies costs: every lane copies its own quad, three window rows and two halos of
 * each population through L1 (four times the bytes the level holds), and three populations
 * ahead is all that fits. Here a block of seven consumer warps and one producer warp takes
 * units of up to seven rows of one set in a 128-column tile. The producer streams the
 * unit's planes (boxes of 136 columns, the two halo rows on either side included)
 * and its carried moments into a ring of shared-memory stages with cp.async.bulk.tensor,
 * tile_stages() populations ahead and on into the next units; a consumer warp has one row, a
 * quad of nodes per lane, and reads own values, window rows and halos from the stage, which
 * the unit's rows share. Stages are guarded by full / empty mbarriers; a consumer releases a
 * stage as soon as its values are in registers. Units come from one counter, the long
 * high-order units first.
 *
 * Boundary work is done in the same loop without reading anything back (branches that are
 * the same for a warp): ghost copies are stored with the value, a shadow's Hermite
 * coefficients are summed as the populations are stored, and a wall row's populations behind
 * the gas-bound ones in population order are kept in shared memory until the fill (the
 * carried moments of a wall row are summed over its final values in order).
 *
 * The arithmetic is layout 9's, operation for operation: the same bits. Two blocks of 256
 * threads per SM, so that one block's epilogue does not leave the SM idle, at 128 registers
 * (FP32 and BF16 still spill 4 to 64 bytes, FP16 none): with an eighth consumer warp (96
 * registers) the loop itself spilled, and with shared memory taking all but 28 KB of L1 each
 * reload went to L2 (1350 cycles a population). Measured
 * (FP32 deviations, us a step, rows of lb_ring2.cuh / tiles): 1024 x 512 Poiseuille 46.8 /
 * 41.9, 1200 x 90 pressure channel 82 / 41; 16384 x 128, whose levels do not fit L2, 97 / 120:
 * the host picks by that (tiles_pay in lb_api.cu).
 *
 * Every wait is bounded; on expiry the block records it in the error word, waits (bounded)
 * for its copies in flight and returns.
 */
#pragma once

#include <cuda_runtime.h>

#include "lb_ring2.cuh"
#include "lb_tma.cuh"
#include "lb_tma.h"

namespace lbk {

constexpr int TILE_COLS = 136, TILE_WARPS = TILE_ROWS;
constexpr int TILE_THREADS = 32 * (TILE_WARPS + 1);
/* a box of the tensor copy must start at a multiple of 128 bytes of shared memory and the
 * rows of a stage follow each other: 4 rows of FP32, 8 of 16-bit values (2176 bytes) */
template <int ST>
__host__ __device__ constexpr int tile_box_bytes() { return tile_box_rows((int)sizeof(typename Store<ST>::T)) * TILE_COLS * (int)sizeof(typename Store<ST>::T); }
template <int ST>
__host__ __device__ constexpr int tile_stage_bytes()
{
    constexpr int B = tile_box_rows((int)sizeof(typename Store<ST>::T));
    static_assert(tile_box_bytes<ST>() % 128 == 0, "alignment of a box");
    return (TILE_ROWS + 4 + B - 1) / B * tile_box_bytes<ST>();
}
/* ring stages: what two blocks per SM leave room for (FP32), more than enough (16-bit) */
template <int ST>
__host__ __device__ constexpr int tile_stages() { return sizeof(typename Store<ST>::T) == 4 ? 11 : 16; }
constexpr int TILE_AUX_BYTES = 3 * TILE_ROWS * 128 * 4;
constexpr int TILE_KEEP_BYTES = 18 * 32 * 16;   /* a top-wall row's values behind the gas-bound ones */
template <int ST>
__host__ __device__ constexpr size_t tile_smem_bytes()
{
    return 128 + (size_t)tile_stages<ST>() * tile_stage_bytes<ST>() + 2 * (TILE_AUX_BYTES + TILE_KEEP_BYTES);
}

/* A consumer's wait: bounded, a few instructions (it stands in every population's body; the
 * error word is written once, by the caller) */
__device__ __forceinline__ bool tile_wait(uint64_t *bar, uint32_t parity)
{
    for (uint32_t n = 0; !mbar_try_wait(bar, parity);)
        if (++n > LB_SPIN_LIMIT) return false;
    return true;
}

/* What a consumer warp carries through the units */
struct TileRing {
    unsigned char *stages;
    uint64_t *full, *empty;
    uint32_t st, parity;   /* the stage to be consumed next */
};

/* One row of set S of Q = n^2 populations (the other set has QT): warp's row w of the unit,
 * lattice row j, lane's quad at x0. GEN: a tile that ends inside, or periodic columns of a
 * width that is not a whole number of quads: stored node by node. Returns false when a wait
 * gave up. */
template <int ST, int Q, int S, int QT, bool COL, bool FORCE, bool GEN>
__device__ __forceinline__ bool tile_row(const StepParams<float> &p, const RingTab &tab, TileRing &rg, const float *aux,
                                         uint64_t *aempty, float4 *keep, int x0, int j, int w, uint8_t flags)
{
    using T = typename Store<ST>::T;
    constexpr int N = Q == 9 ? 3 : (Q == 16 ? 4 : 6);
    constexpr int NH = N * (N / 2);   /* populations bound for one wall */
    constexpr int NS = tile_stages<ST>();
    const int lane = threadIdx.x & 31;
    const RingPop *tp = tab.pop[S];
    const uint32_t plane = (uint32_t)p.plane, pitch = (uint32_t)p.pitch;
    const uint32_t col = (uint32_t)(x0 + LB_GHOST);
    const uint32_t own = (uint32_t)j * pitch + col;
    T *__restrict__ fout = static_cast<T *>(p.fout[S]);
    const float rho0 = p.rho0;
    const float2 nrho02 = f2(-rho0);
    float dl[8];   /* per-column reference density: delta at columns x0 - 2 .. x0 + 5 */
    if constexpr (COL) {
#pragma unroll
        for (int i = 0; i < 8; ++i) dl[i] = (!GEN || x0 < p.nx) ? p.dcol[col - 2 + i] : 0.0f;
    }
    auto dec2 = [&](float2 raw, float2 winv2, int k) -> float2 {
        if constexpr (ST == 1) return fma2(raw, winv2, nrho02);
        else if constexpr (COL) return add2(raw, make_float2(dl[k + 2], dl[k + 3]));
        else return raw;
    };
    auto dec1 = [&](T raw, float winv, int i) -> float {
        if constexpr (COL) return decode_col<ST>(raw, winv, rho0, dl[i]);
        else return decode<ST>(raw, winv, rho0);
    };
    /* boundary work: the wall of a diffuse-wall row (+1 bottom, -1 top, 0 none), the row's
     * ghost-row copies (offsets in rows, 0: none), a quad's periodic image in the ghost
     * columns (its offset; GEN: node by node) and the shadow */
    float wsgn = 0.0f;
    if (j == 0 && p.wall_diffuse[0]) wsgn = 1.0f;
    if (j == p.ny - 1 && p.wall_diffuse[1]) wsgn = -1.0f;
    int img[2] = {0, 0};
    const int nimg = row_images(p, j, img);
    const int im1 = nimg > 0 ? img[0] : 0, im2 = nimg > 1 ? img[1] : 0;
    int img_dx = 0;
    if (p.periodic_x) {
        if (x0 + 3 < LB_GHOST) img_dx = p.nx;
        else if (x0 >= p.nx - LB_GHOST) img_dx = -p.nx;
    }
    const bool shadow = flags & LB_TILE_SHADOW;
    const bool extra = im1 != 0 || img_dx != 0;

    /* four values into row j of a plane (rowp: its storage column 0), its ghost rows and the
     * periodic ghost columns of each */
    auto copies = [&](T *rowp, const T (&e)[4]) {
        auto one = [&](T *r) {
            if constexpr (GEN) {
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (x0 + k < p.nx) put1(p, r, x0 + k, e[k]);
            } else {
                st4(r + col, e);
                if (img_dx != 0) st4(r + col + img_dx, e);
            }
        };
        one(rowp);
        if (im1 != 0) one(rowp + (ptrdiff_t)im1 * (ptrdiff_t)pitch);
        if (im2 != 0) one(rowp + (ptrdiff_t)im2 * (ptrdiff_t)pitch);
    };

    /* 1. the node's coefficients from the carried moments of the level read */
    float2 rd[2], jx[2], jy[2];
    {
        const float4 r4 = *reinterpret_cast<const float4 *>(aux + (0 * TILE_ROWS + w) * 128 + 4 * lane);
        const float4 x4 = *reinterpret_cast<const float4 *>(aux + (1 * TILE_ROWS + w) * 128 + 4 * lane);
        const float4 y4 = *reinterpret_cast<const float4 *>(aux + (2 * TILE_ROWS + w) * 128 + 4 * lane);
        rd[0] = make_float2(r4.x, r4.y);
        rd[1] = make_float2(r4.z, r4.w);
        jx[0] = make_float2(x4.x, x4.y);
        jx[1] = make_float2(x4.z, x4.w);
        jy[0] = make_float2(y4.x, y4.y);
        jy[1] = make_float2(y4.z, y4.w);
        /* the unit's slot is free once every row has its moments (a wall row's also holds what
         * it keeps: see the end) */
        if (wsgn == 0.0f) {
            __syncwarp();
            if (lane == 0) mbar_arrive(aempty);
        }
    }
    const PairNode nd = pair_node_state<FORCE>(p, rd, jx, jy);
    /* the same sums of the values this step stores, and a shadow's second-order ones */
#pragma unroll
    for (int h = 0; h < 2; ++h) rd[h] = jx[h] = jy[h] = f2(0.0f);
    float2 hxx[2], hxy[2], hyy[2];
    float num[4] = {0.0f, 0.0f, 0.0f, 0.0f};   /* wall row: sum over wall-bound |xi.n| w d */
#pragma unroll
    for (int h = 0; h < 2; ++h) hxx[h] = hxy[h] = hyy[h] = f2(0.0f);
    /* deviations as stored, in population order */
    auto sums = [&](const RingPop &rp, const float2 (&ds)[2]) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            rd[h] = fma2(rp.w2, ds[h], rd[h]);
            jx[h] = fma2(rp.wcx2, ds[h], jx[h]);
            jy[h] = fma2(rp.wcy2, ds[h], jy[h]);
        }
        if (shadow) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                hxx[h] = fma2(f2(rp.wxx), ds[h], hxx[h]);
                hxy[h] = fma2(f2(rp.wxy), ds[h], hxy[h]);
                hyy[h] = fma2(f2(rp.wyy), ds[h], hyy[h]);
            }
        }
    };

    /* 2. populations in order, each from the next stage of the ring */
    const int base = ((w + 2) * TILE_COLS + LB_GHOST + 4 * lane) * (int)sizeof(T);
    bool alive = true;
    auto body = [&](auto ac, auto sxc, auto HY, int ystep) {
        const int a = ac;   /* (a compile-time constant for D2Q9) */
        const bool hy = HY;
        constexpr int SXC = decltype(sxc)::value;   /* sign of xi_x; 2: at run time */
        const RingPop &rp = tp[a];
        const int SX = SXC == 2 ? (rp.cx2.x > 0.0f ? 1 : (rp.cx2.x < 0.0f ? -1 : 0)) : SXC;
        if (alive) alive = tile_wait(&rg.full[rg.st], rg.parity);
        const T *sp = reinterpret_cast<const T *>(rg.stages + rg.st * tile_stage_bytes<ST>() + base);
        T own_v[4], yv[3][4], hl[2], hr[2];
        ldn<4>(sp, own_v);
        if (hy) {
            ldn<4>(sp - 2 * ystep, yv[0]);
            ldn<4>(sp - ystep, yv[1]);
            ldn<4>(sp + ystep, yv[2]);
        }
        if (SX != 0) {
            ld2(sp - 2, hl);
            ld2(sp + 4, hr);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&rg.empty[rg.st]);
        if (++rg.st == NS) {
            rg.st = 0;
            rg.parity ^= 1u;
        }
        float2 v[2], c[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) v[h] = dec2(make_float2(to_r(own_v[2 * h]), to_r(own_v[2 * h + 1])), rp.winv2, 2 * h);
        /* collision and force */
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float2 eu;
            if constexpr (SXC == 0) eu = mul2(rp.cy2, nd.uy[h]);
            else eu = fma2(rp.cy2, nd.uy[h], mul2(rp.cx2, nd.ux[h]));
            const float2 t = fma2(mul2(f2(0.5f), eu), eu, eu);
            c[h] = fma2(nd.nom[h], v[h], fma2(nd.P[h], t, nd.B[h]));
            if constexpr (FORCE) c[h] = fma2(nd.dr[h], fma2(rp.gxi2, eu, rp.gxi2), c[h]);
        }
        /* x flux, upwind side by the sign of xi_x */
        if (SX != 0) {
            const float vv[4] = {v[0].x, v[0].y, v[1].x, v[1].y};
            const float winv = rp.winv2.x;
            const float l0 = dec1(hl[0], winv, 0), l1 = dec1(hl[1], winv, 1);
            const float r0 = dec1(hr[0], winv, 6), r1 = dec1(hr[1], winv, 7);
            float Dx[4], d[6], n[6], m[5];
            if (SX > 0) {
                d[0] = l1 - l0;
                d[1] = vv[0] - l1;
                d[2] = vv[1] - vv[0];
                d[3] = vv[2] - vv[1];
                d[4] = vv[3] - vv[2];
                d[5] = r0 - vv[3];
                (void)r1;
            } else {
                d[0] = vv[0] - l1;
                d[1] = vv[1] - vv[0];
                d[2] = vv[2] - vv[1];
                d[3] = vv[3] - vv[2];
                d[4] = r0 - vv[3];
                d[5] = r1 - r0;
                (void)l0;
            }
#pragma unroll
            for (int i = 0; i < 6; ++i) n[i] = neg_part(d[i]);
#pragma unroll
            for (int i = 0; i < 5; ++i) m[i] = minmod_n(d[i], d[i + 1], n[i], n[i + 1]);
#pragma unroll
            for (int k = 0; k < 4; ++k) Dx[k] = fmaf(SX > 0 ? rp.kx : -rp.kx, m[k + 1] - m[k], d[k + 1]);
            c[0] = fma2(rp.ncx2, make_float2(Dx[0], Dx[1]), c[0]);
            c[1] = fma2(rp.ncx2, make_float2(Dx[2], Dx[3]), c[1]);
        }
        /* y flux on the sign-reflected window (rows j - 2s, j - s, j, j + s) */
        if (hy) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float2 w0 = dec2(make_float2(to_r(yv[0][2 * h]), to_r(yv[0][2 * h + 1])), rp.winv2, 2 * h);
                const float2 w1 = dec2(make_float2(to_r(yv[1][2 * h]), to_r(yv[1][2 * h + 1])), rp.winv2, 2 * h);
                const float2 w3 = dec2(make_float2(to_r(yv[2][2 * h]), to_r(yv[2][2 * h + 1])), rp.winv2, 2 * h);
                const float2 d0 = sub2(w1, w0), d1 = sub2(v[h], w1), d2 = sub2(w3, v[h]);
                float2 ma, mb;
                {
                    const float lo = fminf(d1.x, 0.0f), hi = fmaxf(d1.x, 0.0f);
                    ma.x = fminf(fmaxf(d0.x, lo), hi);
                    mb.x = fminf(fmaxf(d2.x, lo), hi);
                }
                {
                    const float lo = fminf(d1.y, 0.0f), hi = fmaxf(d1.y, 0.0f);
                    ma.y = fminf(fmaxf(d0.y, lo), hi);
                    mb.y = fminf(fmaxf(d2.y, lo), hi);
                }
                c[h] = fma2(rp.nacy2, fma2(rp.ky2, sub2(mb, ma), d1), c[h]);
            }
        }
        float2 dn[2], ds[2], e2[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) dn[h] = add2(v[h], c[h]);
        /* as stored, and the deviations the next step would read */
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if constexpr (ST == 1) {
                e2[h] = mul2(rp.w2, add2(f2(rho0), dn[h]));
                ds[h] = fma2(e2[h], rp.winv2, nrho02);
            } else if constexpr (COL) {
                const float2 dc = make_float2(dl[2 * h + 2], dl[2 * h + 3]);
                e2[h] = sub2(dn[h], dc);
                ds[h] = add2(pair_round<ST>(e2[h]), dc);
            } else {
                e2[h] = dn[h];
                ds[h] = pair_round<ST>(dn[h]);
            }
        }
        T *dst = fout + (uint32_t)a * plane + own;
        if (wsgn != 0.0f) {
            const float xn = rp.cy2.x * wsgn;
            if (xn > 0.0f) return;   /* gas-bound: set by the wall below */
            if (xn < 0.0f) {
                const float cw = -xn * rp.w2.x;
                num[0] = fmaf(cw, dn[0].x, num[0]);
                num[1] = fmaf(cw, dn[0].y, num[1]);
                num[2] = fmaf(cw, dn[1].x, num[2]);
                num[3] = fmaf(cw, dn[1].y, num[3]);
            }
        }
        if (wsgn < 0.0f) keep[(a - NH) * 32 + lane] = make_float4(ds[0].x, ds[0].y, ds[1].x, ds[1].y);
        else sums(rp, ds);
        if (!GEN && !extra) {
            pair_st<ST>(dst, e2[0], e2[1]);
        } else {
            const T e[4] = {from_r<T>(e2[0].x), from_r<T>(e2[0].y), from_r<T>(e2[1].x), from_r<T>(e2[1].y)};
            copies(dst - col, e);
        }
    };
    /* D2Q9: nine bodies, each of its abscissae; larger sets: the abscissae of xi_x unrolled (four
     * or six bodies, signs and strides at compile time), rolled over those of xi_y; the few
     * general rows one body, rolled. Instructions are what the kernel waits for most after its
     * stages (2.5 cycles per issue on the 16384 x 128 channel). */
    if constexpr (GEN) {
#pragma unroll 1
        for (int a = 0; a < Q; ++a) {
            const int sy = gh_sign(N, a / N);
            body(a, std::integral_constant<int, 2>{}, sy != 0, sy < 0 ? -TILE_COLS : TILE_COLS);
        }
    } else if constexpr (N == 3) {
        [&]<int... A>(std::integer_sequence<int, A...>) {
            (body(std::integral_constant<int, A>{}, std::integral_constant<int, gh_sign(N, A % N)>{},
                  std::bool_constant<gh_sign(N, A / N) != 0>{}, A / N == 0 ? -TILE_COLS : TILE_COLS),
             ...);
        }(std::make_integer_sequence<int, Q>{});
    } else {
#pragma unroll 1
        for (int iy = 0; iy < N; ++iy) {
            const int ys = iy < N / 2 ? -TILE_COLS : TILE_COLS;
            [&]<int... I>(std::integer_sequence<int, I...>) {
                (body(iy * N + I, std::integral_constant<int, gh_sign(N, I)>{}, std::true_type{}, ys), ...);
            }(std::make_integer_sequence<int, N>{});
        }
    }

    /* 3. diffuse wall (Sec. 3.2): f = rho_W S(u_W) for the gas-bound populations, zero net
     * mass flux through the wall node */
    {
        T *const frow = fout + (size_t)j * pitch;
        if (wsgn != 0.0f) {
            const int wall = wsgn > 0.0f ? 0 : 1;
            const float uwx = p.uw_x[wall], uwy = p.uw_y[wall];
            const float usw = uwx * uwx + uwy * uwy;
            const float kd = p.kdiff[S][wall], kout = p.kout[S][wall];
            float rwd[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) rwd[k] = fmaf(rho0, kd, num[k]) / kout;   /* rho_W - rho0 */
            const int ag = wall == 0 ? Q - NH : 0;
#pragma unroll 1
            for (int i = 0; i < NH; ++i) {
                const RingPop &rp = tp[ag + i];
                const float ew = rp.cx2.x * uwx + rp.cy2.x * uwy;
                const float sm1 = ew + 0.5f * (ew * ew - usw);    /* S / w - 1 */
                T e[4];
                float d[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float dv = fmaf(rwd[k] + rho0, sm1, rwd[k]);
                    if constexpr (COL) {
                        e[k] = encode_col<ST>(dv, rp.w2.x, rho0, dl[k + 2]);
                        d[k] = decode_col<ST>(e[k], rp.winv2.x, rho0, dl[k + 2]);
                    } else {
                        e[k] = encode<ST>(dv, rp.w2.x, rho0);
                        d[k] = decode<ST>(e[k], rp.winv2.x, rho0);
                    }
                }
                copies(frow + (size_t)(ag + i) * plane, e);
                const float2 ds[2] = {make_float2(d[0], d[1]), make_float2(d[2], d[3])};
                sums(rp, ds);
            }
            if (wall == 1) {
                __syncwarp();
#pragma unroll 1
                for (int a = NH; a < Q; ++a) {
                    const float4 q = keep[(a - NH) * 32 + lane];
                    const float2 ds[2] = {make_float2(q.x, q.y), make_float2(q.z, q.w)};
                    sums(tp[a], ds);
                }
            }
        }
    }
    if (!GEN || x0 < p.nx) {
        float *aout = static_cast<float *>(p.aux_out);
        const size_t ap = (size_t)pitch * p.ny;
        const uint32_t m = (uint32_t)j * pitch + (uint32_t)x0;
        __stcg(reinterpret_cast<float4 *>(aout + m), make_float4(rd[0].x, rd[0].y, rd[1].x, rd[1].y));
        __stcg(reinterpret_cast<float4 *>(aout + ap + m), make_float4(jx[0].x, jx[0].y, jx[1].x, jx[1].y));
        __stcg(reinterpret_cast<float4 *>(aout + 2 * ap + m), make_float4(jy[0].x, jy[0].y, jy[1].x, jy[1].y));
    }
    /* 4. mode B: the nodes as the other set's readers see them (hermite_rebuild, term by term) */
    if (shadow) {
        const RingPop *tq = tab.pop[1 - S];
        T *const trow = static_cast<T *>(p.fout[1 - S]) + (size_t)j * pitch;
#pragma unroll 1
        for (int b = 0; b < QT; ++b) {
            const RingPop &rb = tq[b];
            T e[4];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                float2 v = fma2(jx[h], rb.cx2, rd[h]);
                v = fma2(jy[h], rb.cy2, v);
                v = fma2(hxx[h], f2(rb.hxx), v);
                v = fma2(hxy[h], f2(rb.hxy), v);
                v = fma2(hyy[h], f2(rb.hyy), v);
                const float vk[2] = {v.x, v.y};
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    if constexpr (COL) e[2 * h + k] = encode_col<ST>(vk[k], rb.w2.x, rho0, dl[2 * h + k + 2]);
                    else e[2 * h + k] = encode<ST>(vk[k], rb.w2.x, rho0);
                }
            }
            copies(trow + (size_t)b * plane, e);
        }
    }
    if (wsgn != 0.0f) {
        __syncwarp();
        if (lane == 0) mbar_arrive(aempty);
    }
    return alive;
}

/* A unit's stages passed over by a warp without a row in it. Every lane has seen a stage full
 * before lane 0 releases it: once all warps have, the producer refills the stage and its
 * barrier moves on, and a lane still polling would wait on a parity that has gone by. */
template <int ST>
__device__ __forceinline__ bool tile_skip(TileRing &rg, int q)
{
    bool alive = true;
    for (int a = 0; a < q && alive; ++a) {
        alive = tile_wait(&rg.full[rg.st], rg.parity);
        __syncwarp();
        if ((threadIdx.x & 31) == 0) mbar_arrive(&rg.empty[rg.st]);
        if (++rg.st == (uint32_t)tile_stages<ST>()) {
            rg.st = 0;
            rg.parity ^= 1u;
        }
    }
    return alive;
}

/* units[k]: (tile, first row, rows | general << 8, set); sets of 9 (set 0) and Q1
 * populations; ctr[0] the next unit, ctr[1] the blocks that are done (both zero between
 * launches, every launch leaves them so). Odd steps take the units of each kind in the
 * opposite order (the n1 high-order units first in either): what a step wrote last is read
 * first by the next, from L2. */
template <int ST, bool COL, bool FORCE, int Q1>
__global__ void __launch_bounds__(TILE_THREADS, 2)
    tile_kernel(const __grid_constant__ StepParams<float> p, const __grid_constant__ RingTab tab,
                const __grid_constant__ TileMaps maps, const int4 *__restrict__ units, int nunits, int n1,
                uint32_t *__restrict__ ctr, int *__restrict__ err)
{
    extern __shared__ __align__(128) unsigned char tile_raw[];
    constexpr int NS = tile_stages<ST>();
    __shared__ uint64_t full[NS], empty[NS], afull[2], aempty[2];
    __shared__ int4 desc[2];
    unsigned char *sm = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(tile_raw) + 127) & ~(uintptr_t)127);
    unsigned char *aux = sm + NS * tile_stage_bytes<ST>();
    float4 *keep = reinterpret_cast<float4 *>(aux + 2 * TILE_AUX_BYTES);
    const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int k = 0; k < NS; ++k) {
            mbar_init(&full[k], 1);
            mbar_init(&empty[k], TILE_WARPS);
        }
        for (int k = 0; k < 2; ++k) {
            mbar_init(&afull[k], 1);
            mbar_init(&aempty[k], TILE_WARPS);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (warp == TILE_WARPS) {
        /* producer */
        if (lane == 0) {
            uint32_t st = 0, parity = 1, seq = 0;   /* waits on a fresh barrier's parity 1 pass at once */
            bool ok = true;
            uint32_t t = atomicAdd(ctr, 1u);
            for (;;) {
                const bool end = t >= (uint32_t)nunits;
                const uint32_t slot = seq & 1u;
                ok = mbar_wait(&aempty[slot], ((seq >> 1) & 1u) ^ 1u, err, 2);
                if (!ok) break;
                if (end) {
                    desc[slot] = make_int4(-1, 0, 0, 0);
                    mbar_arrive(&afull[slot]);
                    break;
                }
                int k = (int)t;
                if (p.step_key & 1u) k = k < n1 ? n1 - 1 - k : nunits - 1 - (k - n1);
                const int4 u = units[k];
                t = atomicAdd(ctr, 1u);
                desc[slot] = u;
                mbar_arrive_expect_tx(&afull[slot], TILE_AUX_BYTES);
                tma_load_3d(aux + slot * TILE_AUX_BYTES, &maps.aux, &afull[slot], u.x * LB_TILE_X, u.y, 0);
                constexpr int BR = tile_box_rows((int)sizeof(typename Store<ST>::T));
                const int nb = ((u.z & 0xff) + 4 + BR - 1) / BR;
                const int q = u.w ? Q1 : 9;
                const CUtensorMap *map = u.w ? &maps.box[1] : &maps.box[0];
                for (int a = 0; a < q; ++a) {
                    ok = mbar_wait(&empty[st], parity, err, 2);
                    if (!ok) break;
                    mbar_arrive_expect_tx(&full[st], (uint32_t)(nb * tile_box_bytes<ST>()));
                    for (int b = 0; b < nb; ++b)
                        tma_load_3d(sm + st * tile_stage_bytes<ST>() + b * tile_box_bytes<ST>(), map, &full[st], u.x * LB_TILE_X,
                                    u.y + b * BR, a);
                    if (++st == NS) {
                        st = 0;
                        parity ^= 1u;
                    }
                }
                if (!ok) break;
                ++seq;
            }
            if (!ok) {
                /* a consumer gave up: let every copy in flight land (bounded) before the block's
                 * shared memory goes away */
                for (int k = 0; k < NS; ++k) {
                    /* a stage's last copy completes the phase its parity names; an idle one passes */
                    const uint32_t ph = (uint32_t)k < st ? parity ^ 1u : parity;
                    for (uint32_t n = 0; n < LB_SPIN_LIMIT && !mbar_try_wait(&full[k], ph); ++n) {}
                }
                for (uint32_t s = 0; s < 2; ++s) {
                    const uint32_t used = (seq + 2u - s) >> 1;   /* units put in slot s so far, this one included or not */
                    for (uint32_t n = 0; n < LB_SPIN_LIMIT && used > 0 && !mbar_try_wait(&afull[s], (used - 1u) & 1u); ++n) {}
                }
            }
            /* the last block out zeroes the counters for the next launch */
            __threadfence();
            if (atomicAdd(ctr + 1, 1u) == gridDim.x - 1u) {
                ctr[0] = ctr[1] = 0u;
                __threadfence();
            }
        }
        return;
    }
    /* consumers */
    TileRing rg{sm, full, empty, 0u, 0u};
    for (uint32_t seq = 0;; ++seq) {
        const uint32_t slot = seq & 1u;
        if (!mbar_wait(&afull[slot], (seq >> 1) & 1u, err, 1)) return;
        const int4 u = desc[slot];
        if (u.x < 0) return;
        const int s = u.w, nr = u.z & 0xff;
        bool alive = true;
        if (warp < nr) {
            const int j = u.y + warp, x0 = u.x * LB_TILE_X + 4 * lane;
            const uint8_t flags = p.tmap[(size_t)j * p.ntx + u.x];
            const float *ax = reinterpret_cast<const float *>(aux + slot * TILE_AUX_BYTES);
            float4 *kp = keep + slot * (TILE_KEEP_BYTES / 16);
            uint64_t *ae = &aempty[slot];
            const bool gen = u.z >> 8;
            if (s == 0) {
                if (gen) alive = tile_row<ST, 9, 0, Q1, COL, FORCE, true>(p, tab, rg, ax, ae, kp, x0, j, warp, flags);
                else alive = tile_row<ST, 9, 0, Q1, COL, FORCE, false>(p, tab, rg, ax, ae, kp, x0, j, warp, flags);
            } else {
                if (gen) alive = tile_row<ST, Q1, 1, 9, COL, FORCE, true>(p, tab, rg, ax, ae, kp, x0, j, warp, flags);
                else alive = tile_row<ST, Q1, 1, 9, COL, FORCE, false>(p, tab, rg, ax, ae, kp, x0, j, warp, flags);
            }
            __syncwarp();
            /* the pressure columns of this row, once its nodes are stored (see lb_ring2.cuh) */
            if constexpr (!FORCE) {
                if (alive && u.x == 0 && p.pressure[0]) pressure_row<ST>(p, j, 0);
                if (alive && u.x == p.ntx - 1 && p.pressure[1]) pressure_row<ST>(p, j, 1);
            }
        } else {
            __syncwarp();   /* every lane has its copy of the unit: the slot may be refilled */
            if (lane == 0) mbar_arrive(&aempty[slot]);
            alive = tile_skip<ST>(rg, s ? Q1 : 9);
        }
        if (!alive) {
            if (lane == 0) atomicExch(err, 1);
            return;
        }
    }
}

template <int ST, bool COL, bool FORCE, int Q1>
int tile_launch(const StepParams<float> &p, const RingTab &tab, const TileMaps &maps, const int4 *units, int nunits, int n1,
                uint32_t *ctr, int *err, cudaStream_t st)
{
    constexpr size_t smem = tile_smem_bytes<ST>();
    /* per device: the raised shared-memory limit and the resident blocks of the GPU */
    static std::atomic<int> resident[64];
    int dev = 0;
    cudaGetDevice(&dev);
    dev &= 63;
    int nb = resident[dev].load();
    auto kern = tile_kernel<ST, COL, FORCE, Q1>;
    if (nb == 0) {
        int per_sm = 0, nsm = 0;
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, TILE_THREADS, smem) != cudaSuccess ||
            cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || per_sm < 1) {
            cudaGetLastError();
            return -1;
        }
        nb = per_sm * nsm;
        resident[dev].store(nb);
    }
    if (nunits < 1) return 0;
    kern<<<std::min(nb, nunits), TILE_THREADS, smem, st>>>(p, tab, maps, units, nunits, n1, ctr, err);
    return 0;
}

/* layout 10 on tiles for one storage format and high-order set size */
template <int ST, int Q1>
int launch_tiles_store(const StepParams<float> &p, const RingTab &tab, const TileMaps &maps, const int4 *units, int nunits,
                       int n1, uint32_t *ctr, int *err, void *stream)
{
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if constexpr (Store<ST>::dev) {
        if (p.dcol)
            return p.has_force ? tile_launch<ST, true, true, Q1>(p, tab, maps, units, nunits, n1, ctr, err, st)
                               : tile_launch<ST, true, false, Q1>(p, tab, maps, units, nunits, n1, ctr, err, st);
    }
    return p.has_force ? tile_launch<ST, false, true, Q1>(p, tab, maps, units, nunits, n1, ctr, err, st)
                       : tile_launch<ST, false, false, Q1>(p, tab, maps, units, nunits, n1, ctr, err, st);
}

}  // namespace lbk
