"""Plans of the resident steps (res_plan_build, host code) fit the shared memory that a block can
be given: the kernels of one-block parts hold a word of static shared memory beside the plan, and
both together may not pass 227 KB. Compiled against the library on the host; no GPU."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1007_4895_gb300", "csrc")

BLOCK = 227 * 1024   # shared memory of one block, static and dynamic
STATIC = 16          # of it static in the one-block kernels (ptxas -v)

MAIN = r"""
#include <cstdio>
#include <cstdlib>
#include <deque>
#include "lb_internal.h"
using namespace lbk;

struct Rows { std::deque<std::vector<uint8_t>> keep; };

/* a channel of diffuse walls with `rows` high-order rows beside each: tile flags as lb_create's */
static ResLattice channel(Rows &k, int W, int ny, int rows)
{
    std::vector<uint8_t> f(ny, 0);
    auto hi = [&](int j) { return j < rows || j >= ny - rows; };
    for (int j = 0; j < ny; ++j) {
        f[j] = hi(j) ? LB_TILE_HIGH : 0;
        for (int d = -2; d <= 2; ++d)
            if (j + d >= 0 && j + d < ny && hi(j + d) != hi(j)) f[j] |= LB_TILE_SHADOW;
    }
    k.keep.push_back(f);
    return ResLattice{W, ny, {9, 36}, false, {true, true}, k.keep.back().data(), 1, 1};
}

/* one:   W ny rows store        -> smem (0: no plan)
 * sweep: n seed lo hi store     -> smem of a bundle plan of n 8-wide channels */
int main(int argc, char **argv)
{
    for (char line[256]; std::fgets(line, sizeof(line), stdin);) {
        int a, b, c, d, e = 0, cl = 1;
        Rows keep;
        std::vector<ResLattice> L;
        int store = 0;
        if (std::sscanf(line, "one %d %d %d %d %d", &a, &b, &c, &d, &cl) >= 4) {
            L.push_back(channel(keep, a, b, c));
            store = d;
        } else if (std::sscanf(line, "sweep %d %d %d %d %d", &a, &b, &c, &d, &e) == 5) {
            uint32_t s = (uint32_t)b;
            for (int i = 0; i < a; ++i) {
                s = s * 1664525u + 1013904223u;
                const int ny = c + (int)((s >> 8) % (uint32_t)(d - c + 1));
                L.push_back(channel(keep, 8, ny, std::max(2, (15 * ny + 50) / 100)));
            }
            store = e;
        } else {
            return 2;
        }
        ResPlan p;
        const bool pair = store != 0;
        const bool ok = res_plan_build(L, store, pair, cl, 152, 0, p);
        std::printf("%zu %d\n", ok ? p.smem : (size_t)0, ok ? p.parts : 0);
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def plan(tmp_path_factory):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1007_4895_gb300 as lb
    d = tmp_path_factory.mktemp("plan")
    src, exe = str(d / "plan.cpp"), str(d / "plan")
    with open(src, "w") as f:
        f.write("#include <algorithm>\n" + MAIN)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-std=c++20", "-O1", "-I", CSRC, "-I", os.path.join(cuda, "include"), src, "-o", exe,
                    lb.LIB_PATH, "-Wl,-rpath," + os.path.dirname(lb.LIB_PATH)], check=True)

    def run(lines):
        out = subprocess.run([exe], input="\n".join(lines) + "\n", capture_output=True, text=True, check=True).stdout
        return [tuple(int(v) for v in row.split()) for row in out.splitlines()]
    return run


def test_lone_lattices_fit_a_block(plan):
    """Widths and heights around the limit, all storages; at some of them the plan came to exactly
    227 KB, which no launch could be given."""
    cases = [f"one {w} {ny} {rows} {st}" for st in range(5) for w in (4, 5, 8, 12, 13, 16, 31) for rows in (2, 5, 10, 25)
             for ny in range(52, 400, 3)]
    got = plan(cases)
    assert len(got) == len(cases)
    bad = [(c, s) for c, (s, _) in zip(cases, got) if s > BLOCK - STATIC]
    assert not bad, bad[:5]
    assert sum(s > 0 for s, _ in got) > 500 and sum(s == 0 for s, _ in got) > 500


def test_bundles_fit_a_block(plan):
    cases = [f"sweep {n} {seed} 16 {hi} {st}" for st in (1, 2, 4) for hi in (64, 130, 256) for n in (16, 60, 179, 354)
             for seed in range(6)]
    got = plan(cases)
    bad = [(c, s) for c, (s, _) in zip(cases, got) if s > BLOCK - STATIC]
    assert not bad, bad[:5]
    assert sum(parts > 0 for _, parts in got) > len(cases) // 2   # the others hold a channel too tall for a block


def test_cluster_plans_fit_a_block(plan):
    """Kernels on a cluster hold no static shared memory: the whole block is theirs."""
    cases = [f"one {w} {ny} 6 {st} {cl}" for st in (0, 2, 4) for w in (8, 40, 128) for ny in (33, 70, 131, 260) for cl in (2, 4, 8, 16)]
    got = plan(cases)
    assert all(s <= BLOCK for s, _ in got)
    assert sum(s > 0 for s, _ in got) > 20
