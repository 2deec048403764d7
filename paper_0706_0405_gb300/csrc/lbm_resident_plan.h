// lbm_resident_plan.h -- who holds, updates, publishes and receives which
// nodes in the resident kernel (lbm_resident.cu): index arithmetic only, for
// host and device.
//
// A tile is its CTA's own nodes (the core, w x h) with up to `depth` columns
// or rows of other CTAs' nodes around it on the axes that have other CTAs; a
// depth of more than one goes with tiles that span the grid's height (py = 1).
// (c, r) are tile coordinates, (0, 0) the core's first node.  Shell d is what
// lies d columns or rows outside the core: the core after n more steps depends
// on the shells up to n.  All shells are received at an exchange; the j-th of
// the n steps to the next one updates the core and the shells up to n - 1 - j.
#pragma once

#include <stddef.h>

#ifdef __CUDACC__
#define LBM_PLAN_HD __host__ __device__ __forceinline__
#else
#define LBM_PLAN_HD inline
#endif

namespace lbm {

struct ResPlan {
    int px, py;        // CTAs along x and y
    int bw, bh;        // nodes of a core (the last ones along x, y may be smaller)
    int depth;         // steps between exchanges (1 if py > 1)
    int pitch;         // columns per population row of a tile in shared memory
    int cells;         // cells a CTA publishes
    int threads;       // per CTA
    size_t smem;       // dynamic shared memory
    size_t xch_bytes;  // exchange buffer, zeroed by its owner before the first launch
};

// Columns (rows) in shared memory before and after the core: the shells, and
// at least the ghost cell.
LBM_PLAN_HD int res_pad_x(const ResPlan& R) { return R.px > 1 ? R.depth : 1; }
LBM_PLAN_HD int res_pad_y(const ResPlan& R) { return R.py > 1 ? R.depth : 1; }
LBM_PLAN_HD int res_min(int a, int b) { return a < b ? a : b; }
LBM_PLAN_HD int res_max(int a, int b) { return a > b ? a : b; }

struct ResTile {
    int x0, y0, w, h;  // the core
    int l, r, b, t;    // columns and rows of other CTAs' nodes around it
};
LBM_PLAN_HD ResTile res_tile(const ResPlan& R, int nx, int ny, bool perx, bool pery, int cta) {
    ResTile t;
    t.x0 = cta % R.px * R.bw;
    t.y0 = cta / R.px * R.bh;
    t.w = res_min(R.bw, nx - t.x0);
    t.h = res_min(R.bh, ny - t.y0);
    t.l = R.px == 1 ? 0 : perx ? R.depth : res_min(R.depth, t.x0);
    t.r = R.px == 1 ? 0 : perx ? R.depth : res_min(R.depth, nx - t.x0 - t.w);
    t.b = R.py == 1 ? 0 : pery ? R.depth : res_min(R.depth, t.y0);
    t.t = R.py == 1 ? 0 : pery ? R.depth : res_min(R.depth, ny - t.y0 - t.h);
    return t;
}

// Nodes in shell d >= 1.
LBM_PLAN_HD int res_shell(const ResTile& t, int d) {
    return (t.l >= d ? t.h : 0) + (t.r >= d ? t.h : 0) + (t.b >= d ? t.w : 0) + (t.t >= d ? t.w : 0);
}
// The k-th node of the shells 1, 2, ...
LBM_PLAN_HD void res_shell_node(const ResTile& t, int k, int* c, int* r) {
    int d = 1;
    for (int n; k >= (n = res_shell(t, d)); ++d) k -= n;
    int n;
    if (k < (n = t.l >= d ? t.h : 0)) {
        *c = -d, *r = k;
    } else if ((k -= n) < (n = t.r >= d ? t.h : 0)) {
        *c = t.w - 1 + d, *r = k;
    } else if ((k -= n) < (n = t.b >= d ? t.w : 0)) {
        *c = k, *r = -d;
    } else {
        *c = k - n, *r = t.h - 1 + d;
    }
}

// The core's nodes in the order of their update: those that are published
// first (the outer rows and columns on the axes with other CTAs), so that few
// warps publish, then the rest row by row.
LBM_PLAN_HD int res_edge_rows(const ResPlan& R, const ResTile& t) { return R.py > 1 ? res_min(t.h, 2 * R.depth) : 0; }
LBM_PLAN_HD int res_edge_cols(const ResPlan& R, const ResTile& t) { return R.px > 1 ? res_min(t.w, 2 * R.depth) : 0; }
LBM_PLAN_HD int res_edges(const ResPlan& R, const ResTile& t) {
    const int nr = res_edge_rows(R, t);
    return nr * t.w + (t.h - nr) * res_edge_cols(R, t);
}
LBM_PLAN_HD void res_core_node(const ResPlan& R, const ResTile& t, int k, int* c, int* r) {
    const int nr = res_edge_rows(R, t), nc = res_edge_cols(R, t), rh = t.h - nr, rw = t.w - nc;
    const int fr = nr == t.h ? 0 : R.depth, fc = nc == t.w ? 0 : R.depth;  // outer rows, columns on the near side
    if (k < nr * t.w) {
        const int j = k / t.w;
        *r = nr == t.h || j < fr ? j : t.h - nr + j;
        *c = k - j * t.w;
        return;
    }
    k -= nr * t.w;
    const int first = nr > 0 ? fr : 0;  // rows left: first, first + 1, ...
    if (k < rh * nc) {
        const int j = k / rh;
        *c = nc == t.w || j < fc ? j : t.w - nc + j;
        *r = first + k - j * rh;
        return;
    }
    k -= rh * nc;
    *r = first + k / rw;
    *c = (nc > 0 ? fc : 0) + k % rw;
}

constexpr unsigned kNoCell = 0x3fffu;
// Entries to repeat after the edge nodes: where the inner columns are whole
// warps, as many as let the rows begin a warp (whose 32 nodes then lie in 32
// banks).
constexpr int kMaxFill = 31;
LBM_PLAN_HD int res_fill(const ResPlan& R, const ResTile& t) {
    const int inner = t.w - res_edge_cols(R, t);
    const int edges = res_edges(R, t);
    return inner > 0 && inner % 32 == 0 && edges < t.w * t.h ? (32 - edges % 32) % 32 : 0;
}
// The exchange cell of core node (c, r), kNoCell for one that no CTA needs.
LBM_PLAN_HD unsigned res_cell(const ResPlan& R, const ResTile& t, int c, int r) {
    const int n = R.depth;
    int base = 0;
    if (R.py > 1) {
        if (r < n) return (unsigned)(r * R.bw + c);
        if (r >= t.h - n) return (unsigned)((n + r - (t.h - n)) * R.bw + c);
        base = 2 * n * R.bw;
    }
    if (R.px > 1) {
        if (c < n) return (unsigned)(base + c * R.bh + r);
        if (c >= t.w - n) return (unsigned)(base + (n + c - (t.w - n)) * R.bh + r);
    }
    return kNoCell;
}
LBM_PLAN_HD int res_cells(const ResPlan& R) {
    return (R.py > 1 ? 2 * R.depth * R.bw : 0) + (R.px > 1 ? 2 * R.depth * R.bh : 0);
}

// The CTA whose core holds node (c, r) of this tile, and the node's cell there.
LBM_PLAN_HD int res_owner(const ResPlan& R, int nx, int ny, bool perx, bool pery, const ResTile& t, int c, int r,
                          unsigned* cell) {
    const int gx = (t.x0 + c + nx * R.depth) % nx, gy = (t.y0 + r + ny * R.depth) % ny;
    const int cta = gy / R.bh * R.px + gx / R.bw;
    const ResTile o = res_tile(R, nx, ny, perx, pery, cta);
    *cell = res_cell(R, o, gx - o.x0, gy - o.y0);
    return cta;
}

// Whether a tile's rows wrap around inside it: its bottom row's neighbour below
// is its top row.
LBM_PLAN_HD bool res_wraps(const ResPlan& R, bool pery) { return R.py == 1 && pery; }

// Ghost cells of the tile: beside the nodes at a physical side, or at both
// ends of a periodic x axis that the tile spans.
struct ResGhosts {
    int w, e, s, n;  // on the left, right, bottom, top side
};
LBM_PLAN_HD ResGhosts res_ghosts(const ResPlan& R, int nx, int ny, bool perx, bool pery, const ResTile& t) {
    const bool ax = R.px == 1 || !perx, ay = !pery;
    const int n = R.depth, eh = t.h + t.b + t.t, ew = t.w + t.l + t.r;
    ResGhosts g;
    g.w = ax && t.x0 < (R.px == 1 ? 1 : n) ? eh : 0;
    g.e = ax && nx - t.x0 - t.w < (R.px == 1 ? 1 : n) ? eh : 0;
    g.s = ay && t.y0 < (R.py == 1 ? 1 : n) ? ew : 0;
    g.n = ay && ny - t.y0 - t.h < (R.py == 1 ? 1 : n) ? ew : 0;
    return g;
}
struct ResGhost {
    int side, c, r, sc, sr, along;  // the cell, the node it is made from, the node's place along the side
};
LBM_PLAN_HD ResGhost res_ghost(const ResGhosts& n, int nx, int ny, bool perx, bool pery, const ResTile& t, int k) {
    ResGhost g;
    if (k < n.w + n.e) {
        g.side = k < n.w ? 0 : 1;
        g.r = (k < n.w ? k : k - n.w) - t.b;
        g.c = g.side == 0 ? -t.l - 1 : t.w + t.r;
        g.sc = perx ? (g.side == 0 ? t.w - 1 : 0) : (g.side == 0 ? -t.l : t.w + t.r - 1);
        g.sr = g.r;
        g.along = (t.y0 + g.r + ny * (t.b + 1)) % ny;
    } else {
        k -= n.w + n.e;
        g.side = k < n.s ? 2 : 3;
        g.c = (k < n.s ? k : k - n.s) - t.l;
        g.r = g.side == 2 ? -t.b - 1 : t.h + t.t;
        g.sr = g.side == 2 ? -t.b : t.h + t.t - 1;
        g.sc = g.c;
        g.along = (t.x0 + g.c + nx * (t.l + 1)) % nx;
    }
    return g;
}

// Table sizes: ghost cells, received cells and updated nodes of a tile at most.
LBM_PLAN_HD int res_max_ghosts(const ResPlan& R) {
    return 2 * (R.bw + 2 * res_pad_x(R)) + 2 * (R.bh + 2 * res_pad_y(R));
}
LBM_PLAN_HD ResTile res_full_tile(const ResPlan& R) {
    const int x = R.px > 1 ? R.depth : 0, y = R.py > 1 ? R.depth : 0;
    return ResTile{0, 0, R.bw, R.bh, x, x, y, y};
}
// Nodes of the core and the shells up to d.
LBM_PLAN_HD int res_nodes(const ResTile& t, int d) {
    int n = t.w * t.h;
    for (int q = 1; q <= d; ++q) n += res_shell(t, q);
    return n;
}

}  // namespace lbm
