/*
 * lb_resident.cu -- plans of the resident steps (lb_resident.cuh): which rows a block
 * holds, their slots and neighbours, the split of the work, and the shared-memory layout.
 * Host code only; the kernels are instantiated per storage in lb_resident_*.cu.
 */
#include <algorithm>
#include <cstring>
#include <utility>
#include <vector>

#include "lb_internal.h"
#include "lb_resident_host.h"

namespace lbk {

namespace {

size_t up16(size_t v) { return (v + 15) / 16 * 16; }

struct Piece {
    int lat, j0, j1;   /* rows j0 .. j1 - 1 of a lattice */
};
struct Part {
    std::vector<Piece> own;
    ResHead h{};
    std::vector<ResRow> rows;
    std::vector<ResGRow> grow;
    std::vector<uint16_t> push, shlist;
    std::vector<int> ids;
    /* per set: the halo rows (j, slot) of a cluster's band */
    std::vector<std::pair<int, int>> halo[2];
    int nwall = 0;
    size_t smem = 0;
    double cost = 0.0;
};

struct Sizes {
    int V, esize, rsize;
    bool exact, pair;
};

/* rows, slots and neighbours of a part */
bool layout_part(const std::vector<ResLattice> &L, Part &p, const Sizes &z, bool cluster)
{
    const ResLattice &f = L[p.own[0].lat];
    ResHead &h = p.h;
    h.W = f.W;
    const int upr = (f.W + z.V - 1) / z.V;
    const bool images = z.V > 1 && f.W % z.V != 0;
    h.xoff = images ? 4 : 0;
    h.pitch = images ? 4 * upr + 8 : upr * z.V;
    auto magic = [](int n) { return n > 1 ? (uint32_t)(((1ull << 32) + n - 1) / n) : 0u; };   /* exact to 2^16 */
    h.upr_magic = magic(upr);
    auto flag = [&](int lat, int j) { return L[lat].flags[(size_t)j * L[lat].ntx]; };
    auto set_of = [&](int lat, int j) { return (int)(flag(lat, j) & LB_TILE_HIGH); };
    struct Own {
        int k, j, key;   /* piece, row */
    };
    /* slot of row j of piece k in each set: flat tables (a bundle sweep looks up several
     * hundred thousand rows; ordered maps made the plan of 512 channels 40 ms, these 9 ms) */
    std::vector<size_t> base;
    size_t nall = 0;
    for (const Piece &o : p.own) {
        base.push_back(nall);
        nall += (size_t)L[o.lat].ny;
    }
    std::vector<int> slot[2] = {std::vector<int>(nall, -1), std::vector<int>(nall, -1)};
    int nslot[2] = {0, 0};
    std::vector<Own> own[2];
    h.nwall[0] = h.nwall[1] = 0;
    for (size_t k = 0; k < p.own.size(); ++k) {
        const Piece &o = p.own[k];
        p.ids.push_back(o.lat);
        for (int j = o.j0; j < o.j1; ++j) {
            const bool wall = (j == 0 && L[o.lat].wall[0]) || (j == L[o.lat].ny - 1 && L[o.lat].wall[1]);
            /* the rows with the longest chains first: walls, then shadow rows */
            h.nwall[set_of(o.lat, j)] += wall;
            own[set_of(o.lat, j)].push_back({(int)k, j, wall ? 0 : ((flag(o.lat, j) & LB_TILE_SHADOW) ? 1 : 2)});
        }
    }
    for (int s = 0; s < 2; ++s) {
        std::stable_sort(own[s].begin(), own[s].end(), [](const Own &a, const Own &b) { return a.key < b.key; });
        for (const Own &o : own[s]) slot[s][base[o.k] + o.j] = nslot[s]++;
        h.nrow[s] = (int)own[s].size();
        h.nunit[s] = h.nrow[s] * upr;
        h.unit_magic[s] = magic(h.nunit[s]);
        if (h.nunit[s] * 6 > 0xffff) return false;   /* items of a round */
    }
    int nshadow = 0;
    for (int s = 0; s < 2; ++s)
        for (const Own &o : own[s]) {
            const Piece &pc = p.own[o.k];
            const ResLattice &l = L[pc.lat];
            ResRow r{};
            auto at = [&](int d) -> uint16_t {
                int j = o.j + d;
                if (l.periodic_y) j = (j + l.ny) % l.ny;
                else j = std::max(0, std::min(l.ny - 1, j));
                int &n = slot[s][base[o.k] + j];
                if (n < 0) {
                    n = nslot[s]++;
                    if (j < pc.j0 || j >= pc.j1) p.halo[s].push_back({j, n});
                }
                return (uint16_t)n;
            };
            r.own = (uint16_t)slot[s][base[o.k] + o.j];
            r.m2 = at(-2);
            r.m1 = at(-1);
            r.p1 = at(1);
            r.p2 = at(2);
            r.lat = (uint16_t)o.k;
            r.view = RES_NONE;
            r.wallord = r.shord = RES_NONE;
            r.j = (uint16_t)o.j;
            if (o.j == 0 && l.wall[0]) r.flags |= 1;
            else if (o.j == l.ny - 1 && l.wall[1]) r.flags |= 2;
            if (r.flags & 3) r.wallord = (uint16_t)p.nwall++;
            if (flag(pc.lat, o.j) & LB_TILE_SHADOW) {
                r.flags |= RES_SHADOW;
                r.shord = (uint16_t)nshadow++;
                h.nsh[s] += 1;
                p.shlist.push_back((uint16_t)p.rows.size());
            }
            p.rows.push_back(r);
            p.grow.push_back({pc.lat, o.j});
        }
    /* views live where this part's rows of the other set asked for a slot */
    for (int s = 0; s < 2; ++s)
        for (int k = 0; k < h.nrow[s]; ++k) {
            const int i = (s ? h.nrow[0] : 0) + k;
            const int v = slot[1 - s][base[own[s][k].k] + own[s][k].j];
            if (v < 0) continue;
            if (!(p.rows[i].flags & RES_SHADOW)) return false;   /* a reader without a view */
            p.rows[i].view = (uint16_t)v;
        }
    for (int s = 0; s < 2; ++s) {
        h.nslot[s] = nslot[s];
        if (h.nslot[s] > 60000) return false;
        h.q[s] = f.q[s];
        const int n1 = f.q[s] == 9 ? 3 : (f.q[s] == 16 ? 4 : 6);
        h.n[s] = n1;
        h.nh[s] = n1 * (n1 / 2);
    }
    h.nhmax = std::max(h.nh[0], h.nh[1]);
    h.nlat = (int)p.ids.size();
    if (cluster) p.push.assign(8 * p.rows.size(), RES_NONE);
    return true;
}

/* offsets for `rounds` rounds; the bytes needed */
size_t place_part(Part &p, const Sizes &z, int rounds, size_t pop_bytes, size_t lat_bytes)
{
    ResHead &h = p.h;
    h.rounds = rounds;
    for (int s = 0; s < 2; ++s) {   /* whole abscissa rows, so that a row's planes are adjacent */
        h.kr[s] = (h.n[s] + rounds - 1) / rounds;
        h.K[s] = h.kr[s] * h.n[s];
    }
    const int upr = (h.W + z.V - 1) / z.V;
    size_t o = up16(sizeof(ResHead));
    h.off_rows = (uint32_t)o;
    o = up16(o + p.rows.size() * sizeof(ResRow));
    h.off_push = (uint32_t)o;
    o = up16(o + p.push.size() * 2);
    h.off_shlist = (uint32_t)o;
    o = up16(o + p.shlist.size() * 2);
    h.off_ids = (uint32_t)o;
    o = up16(o + p.ids.size() * 4);
    h.table_bytes = (int)o;
    h.off_grow = (uint32_t)o;   /* in the blob, beyond what is copied */
    h.off_lat = (uint32_t)o;
    o = up16(o + p.ids.size() * lat_bytes);
    h.off_pop = (uint32_t)o;
    o = up16(o + pop_bytes);
    h.off_state = (uint32_t)o;
    o = up16(o + (size_t)(h.nunit[0] + h.nunit[1]) * 5 * z.V * z.rsize);
    h.off_herm = (uint32_t)o;
    o = up16(o + (size_t)(h.nsh[0] + h.nsh[1]) * upr * 6 * z.V * z.rsize);
    h.off_wall = (uint32_t)o;
    if (!z.exact) o = up16(o + (size_t)p.nwall * h.nhmax * upr * z.V * z.rsize);
    for (int s = 0; s < 2; ++s) {
        h.off_plane[s] = (uint32_t)o;
        o = up16(o + (size_t)(h.q[s] + h.K[s]) * h.nslot[s] * h.pitch * z.esize);
    }
    p.smem = o;
    return o;
}

/* abscissa rows per item that give the shortest round on the block's warps: an item costs
 * its populations plus about half of one for its set-up */
void split_part(Part &p)
{
    ResHead &h = p.h;
    const int NW = 16;
    double best = 1e30;
    h.rpg[0] = h.rpg[1] = 1;
    for (int g1 = 1; g1 <= h.kr[1]; ++g1)
        for (int g0 = 1; g0 <= h.kr[0]; ++g0) {
            double t[NW] = {};
            const int u1 = (h.nunit[1] * ((h.kr[1] + g1 - 1) / g1) + 31) / 32, u0 = (h.nunit[0] * ((h.kr[0] + g0 - 1) / g0) + 31) / 32;
            for (int u = 0; u < u1 + u0; ++u) t[u % NW] += 0.5 + (u < u1 ? g1 * h.n[1] : g0 * h.n[0]);
            double mx = 0.0, sum = 0.0;
            for (double v : t) mx = std::max(mx, v), sum += v;
            const double c = mx + 0.02 * sum;
            if (c < best) {
                best = c;
                h.rpg[0] = g0;
                h.rpg[1] = g1;
            }
        }
    p.cost = (double)(h.nunit[1] * h.q[1] + h.nunit[0] * h.q[0]) / 32.0;
}

}  // namespace

bool res_plan_build(const std::vector<ResLattice> &L, int store, bool pair, int cluster, int blocks, int sr, ResPlan &out)
{
    const Sizes z{pair ? 4 : 1, store == 0 ? 8 : (store <= 2 ? 4 : 2), store == 0 ? 8 : 4, store == 2, pair};
    const size_t pop_bytes = (L[0].q[0] + L[0].q[1]) * (pair ? sizeof(RingPop) : 16 * (size_t)z.rsize);
    const size_t lat_bytes = 24 * (size_t)z.rsize, limit = res_smem_limit(cluster > 1);
    std::vector<Part> parts;
    if (cluster > 1) {
        if (L.size() != 1 || cluster > RES_MAX_CLUSTER) return false;
        const ResLattice &l = L[0];
        if (l.ny < 2 * cluster) return false;
        /* bands of rows of nearly equal work, at least two rows each (a halo is two rows of
         * one neighbour) */
        std::vector<double> acc(l.ny + 1, 0.0);
        for (int j = 0; j < l.ny; ++j) acc[j + 1] = acc[j] + l.q[l.flags[(size_t)j * l.ntx] & LB_TILE_HIGH] + 3.0;
        int j0 = 0;
        for (int r = 0; r < cluster; ++r) {
            int j1 = l.ny;
            if (r + 1 < cluster) {
                const double want = acc[l.ny] * (r + 1) / cluster;
                j1 = j0 + 2;
                while (j1 < l.ny - 2 * (cluster - 1 - r) && acc[j1] + 0.5 * (acc[j1 + 1] - acc[j1]) < want) ++j1;
            }
            Part p;
            p.own.push_back({0, j0, j1});
            parts.push_back(p);
            j0 = j1;
        }
    } else {
        /* bundles: most work first, each lattice to the least loaded bundle that has room */
        struct Cost {
            double c;
            size_t bytes;
            int i;
        };
        std::vector<Cost> cs;
        size_t total = 0;
        for (size_t i = 0; i < L.size(); ++i) {
            Part p;
            p.own.push_back({(int)i, 0, L[i].ny});
            if (!layout_part(L, p, z, false)) return false;
            bool fits = false;
            for (int r : {1, 2, 3, 6}) {
                if (place_part(p, z, r, pop_bytes, lat_bytes) <= limit) {
                    fits = true;
                    break;
                }
            }
            if (!fits) return false;
            /* a bundle is sized for three rounds */
            const size_t b = place_part(p, z, 3, pop_bytes, lat_bytes) - up16(sizeof(ResHead)) - up16(pop_bytes);
            cs.push_back({(double)p.h.nunit[1] * p.h.q[1] + (double)p.h.nunit[0] * p.h.q[0], b, (int)i});
            total += b;
        }
        std::stable_sort(cs.begin(), cs.end(), [](const Cost &a, const Cost &b) { return a.c > b.c; });
        const size_t cap = limit - up16(sizeof(ResHead)) - up16(pop_bytes);
        blocks = std::max(1, blocks);
        for (size_t nb = std::min<size_t>(L.size(), blocks * ((total + blocks * cap - 1) / (blocks * cap)));;
             nb = std::min<size_t>(L.size(), nb + blocks)) {
            struct Bin {
                double c = 0.0;
                size_t bytes = 0;
                uint64_t group = 0;
                std::vector<int> l;
            };
            std::vector<Bin> bins(nb);
            bool ok = true;
            for (const Cost &k : cs) {
                Bin *to = nullptr;
                for (Bin &b : bins)
                    if ((b.l.empty() || (b.group == L[k.i].group && L[b.l[0]].W == L[k.i].W && b.bytes + k.bytes <= cap)) &&
                        (!to || b.c < to->c))
                        to = &b;
                if (!to) {
                    ok = false;
                    break;
                }
                to->c += k.c;
                to->bytes += k.bytes;
                to->group = L[k.i].group;
                to->l.push_back(k.i);
            }
            if (!ok && nb < L.size()) continue;
            if (!ok) return false;
            std::stable_sort(bins.begin(), bins.end(), [](const Bin &a, const Bin &b) { return a.c > b.c; });
            for (const Bin &b : bins) {
                if (b.l.empty()) continue;
                Part p;
                for (int i : b.l) p.own.push_back({i, 0, L[i].ny});
                parts.push_back(p);
            }
            break;
        }
    }
    for (Part &p : parts)
        if (!layout_part(L, p, z, cluster > 1)) return false;
    if (cluster > 1) {
        /* who stores which rows where */
        for (size_t r = 0; r < parts.size(); ++r)
            for (int s = 0; s < 2; ++s)
                for (const auto &hl : parts[r].halo[s]) {
                    const int j = hl.first;
                    for (size_t o = 0; o < parts.size(); ++o) {
                        Part &p = parts[o];
                        if (o == r || j < p.own[0].j0 || j >= p.own[0].j1) continue;
                        for (size_t i = 0; i < p.rows.size(); ++i) {
                            if (p.grow[i].j != j) continue;
                            const int own_set = (int)i < p.h.nrow[0] ? 0 : 1;
                            if (own_set != s && !(p.rows[i].flags & RES_SHADOW)) return false;
                            uint16_t *to = &p.push[8 * i + (own_set == s ? 0 : 4)];
                            const int t = to[0] == RES_NONE ? 0 : 1;
                            if (to[2 * t] != RES_NONE) return false;
                            to[2 * t] = (uint16_t)r;
                            to[2 * t + 1] = (uint16_t)hl.second;
                            p.rows[i].flags |= RES_PUSH;
                        }
                    }
                }
    }
    /* one number of rounds for the blocks of a cluster (a round ends with a barrier of
     * all of them); each bundle the fewest that fit */
    for (int r : {1, 2, 3, 6}) {
        bool all = true;
        for (Part &p : parts) {
            if (cluster == 1 && p.h.rounds > 0 && p.smem <= limit) continue;
            all = place_part(p, z, r, pop_bytes, lat_bytes) <= limit && all;
        }
        if (all) break;
    }
    out = ResPlan();
    out.cluster = cluster;
    for (Part &p : parts) {
        if (p.smem > limit) return false;
        split_part(p);
        p.h.sr = sr;
        if (cluster > 1)
            for (size_t r = 0; r < parts.size(); ++r)
                for (int s = 0; s < 2; ++s) {
                    p.h.rank[r].off_plane[s] = parts[r].h.off_plane[s];
                    p.h.rank[r].nslot[s] = parts[r].h.nslot[s];
                }
        out.smem = std::max(out.smem, p.smem);
        out.cost = std::max(out.cost, p.cost);
        const size_t at = out.blob.size();
        out.off.push_back((uint32_t)at);
        out.blob.resize(at + up16(p.h.table_bytes + p.grow.size() * sizeof(ResGRow)), 0);
        unsigned char *b = out.blob.data() + at;
        std::memcpy(b, &p.h, sizeof(ResHead));
        std::memcpy(b + p.h.off_rows, p.rows.data(), p.rows.size() * sizeof(ResRow));
        if (!p.push.empty()) std::memcpy(b + p.h.off_push, p.push.data(), p.push.size() * 2);
        if (!p.shlist.empty()) std::memcpy(b + p.h.off_shlist, p.shlist.data(), p.shlist.size() * 2);
        std::memcpy(b + p.h.off_ids, p.ids.data(), p.ids.size() * 4);
        std::memcpy(b + p.h.off_grow, p.grow.data(), p.grow.size() * sizeof(ResGRow));
    }
    out.off.push_back((uint32_t)out.blob.size());
    out.parts = (int)parts.size();
    return true;
}

namespace {
int resident_store(int store, bool pair, const ResLaunch &a)
{
    switch (store) {
        case 0: return pair ? -1 : launch_resident_store<0, false>(a);
        case 1: return pair ? launch_resident_store<1, true>(a) : -1;
        case 2: return pair ? launch_resident_store<2, true>(a) : -1;
        case 3: return pair ? launch_resident_store<3, true>(a) : launch_resident_store<3, false>(a);
        case 4: return pair ? launch_resident_store<4, true>(a) : launch_resident_store<4, false>(a);
        default: return -1;
    }
}
}  // namespace

int launch_resident(int store, bool pair, bool force, const ResPlan &plan, const void *d_plan, const uint32_t *d_off,
                    const void *params, const RingTab *tabs, int nsteps, int base, uint32_t step0, int advance,
                    unsigned int *queue, const void *osc, int blocks, void *stream)
{
    return resident_store(store, pair, {&plan, d_plan, d_off, params, tabs, nsteps, base, step0, advance, queue, osc, blocks,
                                        force, stream, false});
}

bool resident_fits(int store, bool pair, bool force, const ResPlan &plan)
{
    ResLaunch a{};
    a.plan = &plan;
    a.force = force;
    a.query = true;
    return resident_store(store, pair, a) == 0;
}

}  // namespace lbk
