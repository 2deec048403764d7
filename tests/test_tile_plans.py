"""Index arithmetic of the kernels that keep a level on the chip for several
steps, on the CPU: every value a node update would read is the right node's at
the right step, and every node is stored once (csrc/lbm_resident_plan.h and the
strips of csrc/lbm_batch_plan.h, over random grids, splits and sides)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0706_0405_gb300", "csrc")

# A cell holds the step and the global node of its value; -1 and nx (ny) are
# the ghost cells' places.
RESIDENT = r"""
#include <cstdio>
#include <cstdlib>
#include <set>
#include <utility>
#include <vector>
#include "lbm_resident_plan.h"
using namespace lbm;
struct Val { int step = -1, x = 0, y = 0; };
struct Tile {
    ResTile t; ResGhosts g; std::vector<Val> cur, nxt; std::vector<int> item, halo, from;
    std::vector<unsigned> cell, from_cell;
};
#define CHECK(ok) do { if (!(ok)) { printf("line %d: grid %d x %d, core %d x %d, depth %d, periodic %d %d\n", \
                       __LINE__, nx, ny, R.bw, R.bh, R.depth, perx, pery); return 1; } } while (0)
int main() {
    srand(7);
    for (int trial = 0; trial < 3000; ++trial) {
        const int nx = 1 + rand() % (trial % 3 ? 24 : 90), ny = 1 + rand() % (trial % 2 ? 6 : 24);
        const bool perx = rand() % 2, pery = rand() % 2;
        const int steps = 1 + rand() % 14;
        ResPlan R{};
        R.bw = 1 + rand() % nx, R.bh = 1 + rand() % ny;
        R.px = (nx + R.bw - 1) / R.bw, R.py = (ny + R.bh - 1) / R.bh;
        R.depth = R.py == 1 ? 1 + rand() % 4 : 1;
        R.cells = res_cells(R);
        const int ox = res_pad_x(R), oy = res_pad_y(R), P = R.bw + 2 * ox, N = P * (R.bh + 2 * oy), n = R.px * R.py;
        if (n > 60) continue;
        auto place = [&](int c, int r) { return (r + oy) * P + c + ox; };
        auto inside = [&](int c, int r) { return c >= -ox && c < P - ox && r >= -oy && r < R.bh + oy; };
        const ResTile full = res_full_tile(R);
        std::vector<Tile> T(n);
        std::set<std::pair<int, int>> pairs;
        for (int q = 0; q < n; ++q) {
            Tile& a = T[q];
            const ResTile t = a.t = res_tile(R, nx, ny, perx, pery, q);
            a.cur.resize(N), a.nxt.resize(N);
            std::set<int> seen; std::set<unsigned> cells;
            const int items = res_nodes(t, R.depth - 1), core = t.w * t.h;
            CHECK(items <= res_nodes(full, R.depth - 1));
            for (int k = 0; k < items; ++k) {
                int c, r;
                if (k < core) res_core_node(R, t, k, &c, &r); else res_shell_node(t, k - core, &c, &r);
                const bool own = c >= 0 && c < t.w && r >= 0 && r < t.h;
                const unsigned cell = own ? res_cell(R, t, c, r) : kNoCell;
                CHECK(own == (k < core) && inside(c, r) && seen.insert(place(c, r)).second);
                CHECK(!own || (cell != kNoCell) == (k < res_edges(R, t)));
                CHECK(cell == kNoCell || ((int)cell < R.cells && cells.insert(cell).second));
                a.item.push_back(place(c, r)), a.cell.push_back(cell);
            }
            for (int k = 0; k < res_nodes(t, R.depth) - core; ++k) {
                int c, r; unsigned cell;
                res_shell_node(t, k, &c, &r);
                const int o = res_owner(R, nx, ny, perx, pery, t, c, r, &cell);
                CHECK(inside(c, r) && o >= 0 && o < n && (int)cell < R.cells);
                a.halo.push_back(place(c, r)), a.from.push_back(o), a.from_cell.push_back(cell);
                pairs.insert({q, o});
            }
            a.g = res_ghosts(R, nx, ny, perx, pery, t);
            CHECK(a.g.w + a.g.e + a.g.s + a.g.n <= res_max_ghosts(R));
            for (int r = -res_min(t.b + 1, oy); r <= res_min(t.h + t.t, t.h + oy - 1); ++r)
                for (int c = -res_min(t.l + 1, ox); c <= res_min(t.w + t.r, t.w + ox - 1); ++c) {
                    int x = t.x0 + c, y = t.y0 + r;
                    if (R.px > 1 && perx) x = (x + nx * R.depth) % nx;
                    if (R.py > 1 && pery) y = (y + ny * R.depth) % ny;
                    CHECK(x >= -1 && x <= nx && y >= -1 && y <= ny);
                    a.cur[place(c, r)].step = 0, a.cur[place(c, r)].x = x, a.cur[place(c, r)].y = y;
                }
        }
        for (auto& p : pairs) CHECK(pairs.count({p.second, p.first}));  // who receives also publishes
        std::vector<Val> box((size_t)n * (R.cells + 1));
        int j = R.depth - (1 + rand() % R.depth);
        for (int s = 0; s < steps; ++s) {
            const bool more = s + 1 < steps, publish = more && j == R.depth - 1;
            for (int q = 0; q < n; ++q) {
                Tile& a = T[q];
                const bool wraps = res_wraps(R, pery);
                for (int k = 0; k < res_nodes(a.t, res_min(R.depth - j, steps - s) - 1); ++k) {
                    const int p = a.item[k], r = p / P - oy;
                    const int up = wraps && r == a.t.h - 1 ? -(a.t.h - 1) * P : P, down = wraps && r == 0 ? (a.t.h - 1) * P : -P;
                    const int off[5] = {0, 1, -1, up, down}, dx[5] = {0, 1, -1, 0, 0}, dy[5] = {0, 0, 0, 1, -1};
                    for (int e = 0; e < 5; ++e) {
                        const Val v = a.cur[p + off[e]];
                        int x = a.cur[p].x + dx[e], y = a.cur[p].y + dy[e];
                        if (perx && R.px > 1) x = (x + nx) % nx;
                        if (pery) y = R.py > 1 || wraps ? (y + ny) % ny : y;
                        CHECK(v.step == s && v.x == x && v.y == y);
                    }
                    a.nxt[p] = a.cur[p], a.nxt[p].step = s + 1;
                    if (publish && a.cell[k] != kNoCell) box[(size_t)q * R.cells + a.cell[k]] = a.nxt[p];
                }
            }
            for (int q = 0; q < n; ++q) {
                Tile& a = T[q];
                for (size_t k = 0; k < a.halo.size() && publish; ++k) {
                    const Val v = box[(size_t)a.from[k] * R.cells + a.from_cell[k]];
                    const int c = a.halo[k] % P - ox, r = a.halo[k] / P - oy;
                    CHECK(v.step == s + 1 && v.x == (a.t.x0 + c + nx * R.depth) % nx && v.y == (a.t.y0 + r + ny * R.depth) % ny);
                    a.nxt[a.halo[k]] = v;
                }
                for (int k = 0; k < a.g.w + a.g.e + a.g.s + a.g.n; ++k) {
                    const ResGhost g = res_ghost(a.g, nx, ny, perx, pery, a.t, k);
                    CHECK(inside(g.c, g.r) && inside(g.sc, g.sr));
                    const Val v = a.nxt[place(g.sc, g.sr)];
                    const bool x = g.side < 2;
                    const int far = x ? nx - 1 : ny - 1;
                    if (v.step == s + 1)
                        CHECK(g.along == (x ? v.y : v.x) &&
                              (x ? v.x : v.y) == ((g.side & 1) != (x && perx) ? far : 0));
                    a.nxt[place(g.c, g.r)] = {v.step, x ? (g.side == 0 ? -1 : nx) : v.x, x ? v.y : (g.side == 2 ? -1 : ny)};
                }
                a.cur.swap(a.nxt);
            }
            j = publish ? 0 : j + 1;
        }
    }
    puts("ok");
}
"""

# Columns: the step of each lane's value; a window's outermost lanes go stale
# one by one, and every column is stored once at full age.
STRIPS = r"""
#include <cstdio>
#include <cstdlib>
#include "lbm_batch_plan.h"
using namespace lbm;
#define CHECK(ok) do { if (!(ok)) { printf("line %d, trial %d\n", __LINE__, trial); return 1; } } while (0)
int main() {
    srand(7);
    for (int trial = 0; trial < 600; ++trial) {
        const int np = 1 + rand() % 30, ns = 3 + 2 * (rand() % 3), nw = 4, grid = 1 + rand() % 700;
        std::vector<int> nx(np);
        for (int& x : nx) x = 1 + rand() % (rand() % 4 == 0 ? 8 : rand() % 2 ? 140 : 2000);
        std::vector<StripWarp> plan;
        const int rounds = strip_plan(np, nx.data(), ns, grid, nw, plan);
        CHECK(plan.size() == (size_t)rounds * nw);
        std::vector<std::vector<int>> stored(np);
        for (int p = 0; p < np; ++p) stored[p].assign(nx[p] + 2, 0);
        for (int r = 0; r < rounds; ++r) {
            const StripWarp* W = plan.data() + (size_t)r * nw;
            int age[4][32], next[4][32];
            for (int w = 0; w < nw; ++w) {
                if (W[w].prob < 0) continue;
                const int end = nx[W[w].prob];
                CHECK(W[w].col0 >= -1 && W[w].slot >= 0 && W[w].slot <= w && (end - W[w].col0 >= 32 || end > W[w].col0));
                if (W[w].links & 1) CHECK(w > 0 && (W[w - 1].links & 2) && W[w - 1].prob == W[w].prob &&
                                          W[w - 1].slot == W[w].slot && W[w - 1].col0 + 30 == W[w].col0);
                if (W[w].links & 2) CHECK(w + 1 < nw && (W[w + 1].links & 1));
                for (int l = 0; l < 32; ++l) age[w][l] = W[w].col0 + l <= end ? 0 : -100;
            }
            for (int s = 0; s < ns; ++s) {
                for (int w = 0; w < nw; ++w) {
                    if (W[w].prob < 0) continue;
                    for (int l = 0; l < 32; ++l) {
                        const bool fresh = l > 0 && l < 31 && age[w][l - 1] == s && age[w][l] == s && age[w][l + 1] == s;
                        next[w][l] = fresh ? s + 1 : -100;
                    }
                    const int gr = nx[W[w].prob] - W[w].col0;
                    if (W[w].col0 < 0) next[w][0] = next[w][1];
                    if (gr < 32) next[w][gr] = next[w][gr - 1];
                }
                for (int w = 0; w < nw; ++w) {
                    if (W[w].prob < 0) continue;
                    for (int l = 0; l < 32; ++l) age[w][l] = next[w][l];
                    if (s + 1 < ns && (W[w].links & 1)) age[w][0] = next[w - 1][30];
                    if (s + 1 < ns && (W[w].links & 2)) age[w][31] = next[w + 1][1];
                }
            }
            for (int w = 0; w < nw; ++w) {
                if (W[w].prob < 0) continue;
                const int end = nx[W[w].prob], gr = end - W[w].col0;
                for (int l = 0; l < 32; ++l) {
                    const int c = W[w].col0 + l;
                    const bool mine = c >= W[w].c0 && c < W[w].c1 && !(l == 0 && (W[w].links & 1)) && !(l == 31 && (W[w].links & 2));
                    const bool ghost = (W[w].col0 < 0 && l == 0 && W[w].c0 == 0) || (l == gr && W[w].c1 == end);
                    if (!mine && !ghost) continue;
                    CHECK(age[w][l] == ns);
                    ++stored[W[w].prob][c + 1];
                }
            }
        }
        for (auto& v : stored)
            for (int n : v) CHECK(n == 1);
    }
    puts("ok");
}
"""


@pytest.mark.parametrize("name,source", [("resident", RESIDENT), ("strips", STRIPS)])
def test_every_value_read_is_the_right_nodes(name, source, tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / f"{name}.cpp", tmp_path / name
    src.write_text(source)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout == "ok\n", out.stdout
