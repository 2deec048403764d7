// lbm_batch_plan.h -- host-side planning of the batch kernel's step order
// (plain C++, no CUDA): for each CTA of a launch, the other CTAs whose tiles
// border one of its own, so that a CTA can start step s + 1 as soon as those
// have finished step s.
#pragma once

#include <vector>

namespace lbm {

// Tile t of the batch is tile (ix, iy) of problem p, whose tiles form a
// tiles_x[p] x tiles_y[p] grid numbered from base[p] in row order.  Two tiles
// border each other if they are next to each other in x or y, or if they are
// the first and last tile of a row (column) of a problem with a periodic x
// (y) side.  owner(t) is the CTA that walks tile t.  out receives max_nbr
// entries per CTA, -1 padded; returns false if some CTA borders more than
// max_nbr others (the caller then orders the steps by a grid barrier).
template <class Owner>
bool batch_plan_neighbours(int ntiles, const int* tile_p, const int* tile_ix, const int* tile_iy,
                           const int* tiles_x, const int* tiles_y, const int* base,
                           const unsigned char* periodic_x, const unsigned char* periodic_y, int grid,
                           Owner owner, int max_nbr, std::vector<int>& out) {
    out.assign((size_t)grid * (size_t)max_nbr, -1);
    std::vector<int> cnt((size_t)grid, 0);
    auto add = [&](int c, int n) {
        if (n == c) return true;
        for (int j = 0; j < cnt[(size_t)c]; ++j)
            if (out[(size_t)c * max_nbr + j] == n) return true;
        if (cnt[(size_t)c] == max_nbr) return false;
        out[(size_t)c * max_nbr + cnt[(size_t)c]++] = n;
        return true;
    };
    for (int t = 0; t < ntiles; ++t) {
        const int p = tile_p[t], tx = tiles_x[p], ty = tiles_y[p];
        const int ix = tile_ix[t], iy = tile_iy[t], c = owner(t);
        const int nb[4][2] = {{ix - 1, iy}, {ix + 1, iy}, {ix, iy - 1}, {ix, iy + 1}};
        for (const auto& q : nb) {
            int jx = q[0], jy = q[1];
            if (jx < 0 || jx >= tx) {
                if (!periodic_x[p]) continue;
                jx = (jx + tx) % tx;
            }
            if (jy < 0 || jy >= ty) {
                if (!periodic_y[p]) continue;
                jy = (jy + ty) % ty;
            }
            if (!add(c, owner(base[p] + jy * tx + jx))) return false;
        }
    }
    return true;
}

// ------------------------------------------------------------------ strips
// A warp of the strip kernel (lbm_strip.cu): lane l holds grid column col0 + l
// of problem prob (-1: idle).  Consecutive warps of a window overlap by two
// columns, lane 0 and lane 31 being copies of the neighbours' lanes 30 and 1.
// The window stores the columns [c0, c1) and carries ns more on either side,
// or the ghost column where the problem ends first.  links: bit 0 / 1, the
// window goes on in the previous / next warp.  slot: the window's place among
// the CTA's.
struct StripWarp {
    int prob, col0, c0, c1, links, slot;
};

// Windows of all columns of the problems (nx[p] each) for passes of up to ns
// steps, packed into rounds of `warps` warps; a round is what a CTA advances
// at a time.  out receives `stride` entries a round.  Returns the rounds.
inline int strip_pack(int nprob, const int* nx, int ns, int warps, int stride, std::vector<StripWarp>& out) {
    const StripWarp idle = {-1, 0, 0, 0, 0, 0};
    out.clear();
    int used = warps, slots = 0, rounds = 0;  // no round begun
    for (int p = 0; p < nprob; ++p)
        for (int c0 = 0; c0 < nx[p];) {
            const int g0 = c0 - ns > -1 ? c0 - ns : -1;  // first column of the window
            const int avail = warps - used;
            int need = (nx[p] + 1 - g0 - 2 + 29) / 30;  // 30 columns a warp and two
            if (need < 1) need = 1;
            int c1 = nx[p];
            if (need > avail) {
                need = avail;
                c1 = g0 + 30 * avail + 2 - ns;
                // a short piece at the end of a round is not worth its halo
                if (avail == 0 || (used > 0 && c1 - c0 < 30)) {
                    out.resize((size_t)(++rounds) * stride, idle);
                    used = slots = 0;
                    continue;
                }
            }
            for (int j = 0; j < need; ++j)
                out[(size_t)(rounds - 1) * stride + used + j] = {p, g0 + 30 * j, c0, c1,
                                                                 (j > 0 ? 1 : 0) | (j + 1 < need ? 2 : 0), slots};
            used += need;
            ++slots;
            c0 = c1;
        }
    return rounds;
}

// The packing for a grid of `grid` CTAs of up to max_warps warps: as many
// rounds to a CTA as rounds of max_warps warps give, then the fewest warps a
// round that keep to that number, so that all CTAs work equally long.
inline int strip_plan(int nprob, const int* nx, int ns, int grid, int max_warps, std::vector<StripWarp>& out) {
    const int per = (strip_pack(nprob, nx, ns, max_warps, max_warps, out) + grid - 1) / grid;
    int lo = 1, hi = max_warps;
    while (lo < hi) {
        const int mid = (lo + hi) / 2;
        if (strip_pack(nprob, nx, ns, mid, max_warps, out) <= per * grid) hi = mid;
        else lo = mid + 1;
    }
    return strip_pack(nprob, nx, ns, lo, max_warps, out);
}

}  // namespace lbm
