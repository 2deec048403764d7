// lbm_resident.cu -- several time steps of a small grid in one launch, the
// level held in shared memory (Eq. SEC-VON-11, the same per-node arithmetic
// as the one-step kernels).
//
// A grid of up to a few hundred thousand nodes is bound by launches: a step of
// the tile kernel takes 3.6 to 5.4 us however few nodes it updates (launch,
// tensor map, box copy, drain).  Here each CTA of one cooperative launch owns
// a fixed tile, keeps its level in shared memory for all the steps and
// exchanges only the tile's edge nodes with the CTAs next to it.  Measured, us
// a step, launch a step -> here (FP32_TDF / FP32_CONS / FP32_T64): 400 x 4
// 5.3 -> 1.0 / 3.6 -> 0.9 / 4.5 -> 1.3, 2000 x 4 5.4 -> 1.0 / 3.7 -> 0.9 /
// 4.5 -> 1.4, 400 x 100 6.1 -> 1.8 / 4.7 -> 1.7 / 5.8 -> 2.4, 1024 x 256
// 8.8 -> 4.3 / 7.3 -> 3.8 / 11.4 -> 6.7; FP64: 400 x 4 6.1 -> 2.6,
// 2000 x 4 6.0 -> 3.6.  A small tile's step is a chain of latencies: the node
// update 950 cycles, the exchange about 1300 (of which 1000 from one CTA's
// store to another's poll, measured between neighbours among 50 to 125 CTAs),
// barriers 150; a large one's is issue- and shared-memory-bound.
//  * two copies of the tile with a halo, [row][population][column] like a
//    level; a step reads one and writes the other;
//  * tiles that span the grid's height keep a halo of up to four columns and
//    exchange every fourth step only, updating the columns of the halo that
//    later steps need in between (lbm_resident_plan.h has the index
//    arithmetic); where such a grid is periodic in y, a node at its bottom or
//    top finds the row around the edge in the tile, without ghost cells;
//  * a step is: the threads update the tile's nodes, its edge nodes first,
//    and publish the edge nodes' values from registers as they go; the
//    last warps poll the halo cells, one cell (nine values) a thread, while
//    others fill the tile's ghost cells from tables made at the start; a
//    barrier ends the step, and one before the ghost cells where the tile has
//    any.  (Publishing in a phase of its own after a barrier cost 0.35 us a
//    step; ghost rules and polls in the edge nodes' own threads up to 3600
//    cycles, where the node update takes 900);
//  * edge values travel as 128-bit words of three 32-bit values and the
//    exchange they belong to (FP64: one value), written and polled with
//    relaxed GPU-scope accesses.  The tag makes a word its own flag: no fence,
//    no second round trip.  Slots alternate by the exchange's parity: a CTA
//    publishes exchange t + 2 only after it has received its neighbours'
//    t + 1, which they publish after a barrier that follows their reads of t.  Tags come from a counter in device memory
//    that only grows, advanced by the last CTA to leave, so replays of a
//    captured launch work;
//  * the place of a moving split (the double Mach reflection's top boundary)
//    is turned into an index once a step, by a warp of its own;
//  * the last two steps also write their levels to the context's buffers,
//    ghosts included, so that every call leaves what the one-step kernels
//    would have left.
// Polls are bounded (lbm_batch_set_wait_limit): on give-up the CTA raises
// ST_TIMEOUT and leaves, and so do the others, which watch that word while
// they poll.
#include <climits>

#include "lbm_launch.h"

namespace lbm {

namespace {
// SM cycles a poll lasts before it gives up, ~2 s at 2 GHz (resident_set_wait_cycles)
__device__ long long g_poll_cycles = 4000000000LL;
constexpr int kMaxDepth = 4;  // steps between exchanges at most

__device__ __forceinline__ void st_word(ResWord* p, unsigned a, unsigned b, unsigned c, unsigned tag) {
    asm volatile(
        "{\n\t.reg .b128 t;\n\t.reg .b64 l, h;\n\tmov.b64 l, {%1, %2};\n\tmov.b64 h, {%3, %4};\n\t"
        "mov.b128 t, {l, h};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
        "r"(a), "r"(b), "r"(c), "r"(tag)
        : "memory");
}
__device__ __forceinline__ ResWord ld_word(const ResWord* p) {
    ResWord w;
    asm volatile(
        "{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
        : "=l"(w.lo), "=l"(w.hi)
        : "l"(p)
        : "memory");
    return w;
}
__device__ __forceinline__ unsigned word_tag(const ResWord& w) { return (unsigned)(w.hi >> 32); }

// Words per cell: three FP32 values each, or one FP64 value.
template <typename S>
constexpr int kCellWords = sizeof(S) == 4 ? 3 : 9;

// Modes that repeat a node for the sake of shared-memory banks (res_fill); where
// the FP64 pipe is the bound, a warp more costs 1 %.
template <typename S, int TM>
constexpr bool fills() {
    return sizeof(S) == 4 && TM != T_INT64;
}

// A node's entry in the table of the nodes to update: its place in the tile,
// its exchange cell, and whether the row above (below) it is the bottom (top)
// one of a tile that wraps around.
constexpr unsigned kWrapUp = 1u << 30, kWrapDown = 1u << 31;
__device__ __forceinline__ int item_place(unsigned e) { return (int)(e & 0xffffu); }
__device__ __forceinline__ unsigned item_cell(unsigned e) { return e >> 16 & kNoCell; }

// Values of one node after a step, FP32 modes, from the box b (populations P
// apart, the rows above and below dn and ds away).
template <int TM>
__device__ __forceinline__ unsigned node_update(const Model<float>& M, const float* b, int P, int dn, int ds,
                                                float (&o)[9]) {
    float f[9], rho, ux, uy, T;
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = b[i * P];
    moments<float, TM>(f, M, rho, ux, uy, T);
    relaxation<float, TM>(M, f, rho, ux, uy, T, o);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const float* p = b + i * P;
        o[i] = update(M, i, o[i], f[i], p[1], p[-1], p[dn], p[ds]);
    }
    return health(rho, ux, uy, T);
}
// FP64, four warps to 32 nodes.  An FP64 instruction occupies its SM
// quarter's pipe for 64 cycles whatever the number of active lanes (measured;
// two results per SM and cycle), so a lone warp takes 99 x 64 cycles for its
// nodes.  Here the four warps that share 32 nodes sit on the four quarters and
// split the node update of lbm_fp64.cuh by population pairs, at most 41
// instructions each: warp 0 updates populations 1 and 3, warp 1 the pair 2, 4
// and the rest population, warp 2 the pair 5, 7, warp 3 the pair 6, 8.  Pair
// sums and the moments that every warp needs are formed by one warp each and
// handed over in shared memory (a CTA barrier costs less than one instruction
// of the pipe).  The operations and their order are those of
// fp64_relaxation and fp64_update, so the bits are too.
constexpr int kQuadGroups = 3;  // 32-node groups per CTA at most
__device__ __forceinline__ unsigned quad_update(const Fp64Step& C, const double* cur, double* nxt,
                                                const unsigned* item, int n_items, int P, int around) {
    __shared__ double pairs[kQuadGroups][8][32];  // differences (0..3) and sums (4..7) of the warps' pairs
    __shared__ double mom[kQuadGroups][5][32];    // 1 / rho, rho, gx, gy, E / b
    const int lane = threadIdx.x & 31, role = threadIdx.x / 32 & 3, group = threadIdx.x / 128;
    const int q = group * 32 + lane;
    const bool in = q < n_items;
    const unsigned it = item[in ? q : 0];
    const int at = item_place(it);
    const int dn = it & kWrapUp ? -around : 9 * P, ds = it & kWrapDown ? around : -9 * P;
    const double* b = cur + at;
    // the pair's populations against and along its direction
    const int lo = role == 0 ? 1 : role == 1 ? 2 : role == 2 ? 5 : 8, hi = role == 0 ? 3 : role == 1 ? 4 : role == 2 ? 7 : 6;
    const double fl = b[lo * P], fh = b[hi * P], f0 = b[0];
    pairs[group][role][lane] = fh - fl;
    pairs[group][4 + role][lane] = fl + fh;
    __syncthreads();
    const double(*d)[32] = pairs[group];
    if (role == 0) {
        const double rho = (f0 + (d[4][lane] + d[5][lane])) + (d[6][lane] + d[7][lane]);
        mom[group][0][lane] = fp64_rcp(rho);
        mom[group][1][lane] = rho;
    } else if (role == 1) {
        mom[group][2][lane] = __fma_rn(C.kap, d[2][lane] + d[3][lane], d[0][lane]);
    } else if (role == 2) {
        mom[group][3][lane] = __fma_rn(C.kap, d[2][lane] - d[3][lane], d[1][lane]);
    } else {
        mom[group][4][lane] = fp64_energy(C, f0, d[4][lane] + d[5][lane], d[6][lane] + d[7][lane]);
    }
    __syncthreads();
    const double inv = mom[group][0][lane], rho = mom[group][1][lane], gx = mom[group][2][lane],
                 gy = mom[group][3][lane];
    const double Ux = gx * inv, Uy = gy * inv;
    const double xx = gx * Ux, yy = gy * Uy, qq = xx + yy;
    const double p = __fma_rn(-C.t1, qq, mom[group][4][lane]);
    const double V = __fma_rn(C.vp, p, qq) * inv;
    double B, sum, g;
    if (role < 2) {
        const double A = __fma_rn(C.a1p, p, __fma_rn(C.a1q, qq, C.a1r * rho));
        B = __fma_rn(C.b1v, V, C.b1c);
        sum = __fma_rn(C.h1, role == 0 ? xx : yy, A);
        g = role == 0 ? gx : gy;
    } else {
        const double A = __fma_rn(C.a5p, p, __fma_rn(C.a5q, qq, C.a5r * rho));
        B = __fma_rn(C.b5v, V, C.b5c);
        sum = __fma_rn(role == 2 ? C.k5 : -C.k5, gx * Uy, A);
        g = role == 2 ? gx + gy : gx - gy;
    }
    if (!in) return 0u;
    auto store = [&](int i, double r, double c) {
        const double* n = b + i * P;
        nxt[at + i * P] = fp64_update(C, i, r, c, n[1], n[-1], n[dn], n[ds]);
    };
    store(lo, __fma_rn(-B, g, sum), fl);
    store(hi, __fma_rn(B, g, sum), fh);
    if (role == 1) store(0, C.k0 * p, f0);
    return fp64_health(rho, p, V);
}

// First along-side index in the "hi" part of a side at time level `level`:
// the same decision as side_part for every index, since (j + 1/2) dx does not
// decrease with j.
template <typename S>
__device__ __forceinline__ int split_at(const Grid<S>& G, int side, long long level) {
    if (!G.split_moving[side]) return G.split_index[side];
    const int len = side < S_BOTTOM ? G.ny : G.nx;
    const double t = __dmul_rn((double)level, G.dt);
    const double split = __dadd_rn(G.split0[side], __dmul_rn(G.split_speed[side], t));
    const float guess = (float)split / (float)G.dx;
    int j = guess > 0.0f ? (guess < (float)len ? (int)guess : len) : 0;
    while (j < len && __dmul_rn((double)j + 0.5, G.dx) < split) ++j;
    while (j > 0 && !(__dmul_rn((double)(j - 1) + 0.5, G.dx) < split)) --j;
    return j;
}

// Fill one ghost cell of a tile (the rules of write_ghosts): g and src are
// population 0 of the ghost cell and of the node it is made from, P apart.
template <typename S>
__device__ __forceinline__ void fill_ghost(const Grid<S>& G, int side, int part, S* g, const S* src, int P) {
    const int kind = part ? G.kind_hi[side] : G.kind_lo[side];
    S v[9];
    if (kind == BC_DIRICHLET) {
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = G.feq[side][part][i];
    } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = src[i * P];
    }
    if (kind == BC_REFLECT) {
        // population i of the ghost cell is the mirror one's value: store
        // where the mirror map sends it (it is its own inverse)
        const bool x = side < S_BOTTOM;
#pragma unroll
        for (int i = 0; i < 9; ++i) g[(x ? mirror_x(i) : mirror_y(i)) * P] = v[i];
    } else {
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i * P] = v[i];
    }
}

// Poll the words of one halo cell until all carry the tag, and put the nine
// values at dst (P apart).  False if the poll gave up.
template <typename S>
__device__ __forceinline__ bool receive(const ResWord* src, unsigned tag, S* dst, int P, const unsigned* status) {
    constexpr int Q = kCellWords<S>;
    ResWord w[Q];
    long long t0 = 0;
    for (unsigned spins = 0;; ++spins) {
#pragma unroll
        for (int k = 0; k < Q; ++k) w[k] = ld_word(src + k);
        unsigned miss = 0;
#pragma unroll
        for (int k = 0; k < Q; ++k) miss |= word_tag(w[k]) ^ tag;
        if (miss == 0) break;
        if ((spins & 63) == 63) {
            const long long t = clock64();
            if (t0 == 0) t0 = t;
            if (t - t0 > g_poll_cycles || (*(volatile const unsigned*)status & ST_TIMEOUT)) return false;
        }
    }
#pragma unroll
    for (int k = 0; k < Q; ++k) {
        if constexpr (sizeof(S) == 4) {
            dst[(3 * k) * P] = __uint_as_float((unsigned)w[k].lo);
            dst[(3 * k + 1) * P] = __uint_as_float((unsigned)(w[k].lo >> 32));
            dst[(3 * k + 2) * P] = __uint_as_float((unsigned)w[k].hi);
        } else {
            dst[k * P] = __longlong_as_double((long long)w[k].lo);
        }
    }
    return true;
}
}  // namespace

// FP32: one node a thread in rounds of the CTA's threads, no barrier between
// them (a thread of two nodes in packed arithmetic was no faster at any size:
// one CTA per SM has to overlap its own warps' shared-memory and arithmetic
// phases, which wants many small items).  FP64: four warps to 32 nodes,
// quad_update.  sync: [0] the tag counter, [1] CTAs that have left (zero
// between launches).
template <typename S, int TM, int kThreads, typename C>
__global__ void __launch_bounds__(kThreads, 1)
    k_resident(const __grid_constant__ C M, const __grid_constant__ Grid<S> G, const __grid_constant__ ResPlan R,
               const __grid_constant__ ResRun<S> A) {
    extern __shared__ __align__(16) unsigned char smem[];
    const int P = R.pitch, RS = 9 * R.pitch;
    const int T = blockDim.x, tid = threadIdx.x, cta = blockIdx.x;
    const bool perx = G.kind_lo[S_LEFT] == BC_PERIODIC, pery = G.kind_lo[S_BOTTOM] == BC_PERIODIC;
    const ResTile t = res_tile(R, G.nx, G.ny, perx, pery, cta);
    const int x0 = t.x0, y0 = t.y0, w = t.w, h = t.h;
    const int pad_x = res_pad_x(R), pad_y = res_pad_y(R);
    const size_t buf = (size_t)(R.bh + 2 * pad_y) * RS;
    S* cur = reinterpret_cast<S*>(smem);
    S* nxt = cur + buf;
    // tables: per ghost cell its place, its source's, its side and along-side
    // index; per received cell its source's; per node its place and the cell
    // it is published as; per received cell its place
    const ResTile full = res_full_tile(R);
    const int max_halo = res_nodes(full, R.depth) - R.bw * R.bh;
    uint2* ghost = reinterpret_cast<uint2*>(nxt + buf);
    unsigned* halo_src = reinterpret_cast<unsigned*>(ghost + res_max_ghosts(R));
    unsigned* item = halo_src + max_halo;
    unsigned short* halo_dst = reinterpret_cast<unsigned short*>(item + res_nodes(full, R.depth - 1) + kMaxFill);
    __shared__ int split_now[2][4];  // by the step's parity
    __shared__ int upto[kMaxDepth];  // nodes of the core and the shells up to d
    const int origin = pad_y * RS + pad_x;  // node (0, 0), population 0, in a buffer
    const unsigned epoch = *(volatile unsigned*)A.sync;
    const size_t pl = (size_t)G.plane;

    const bool wraps = res_wraps(R, pery);
    const int around = (h - 1) * RS;  // from the bottom row to the top row
    // (fills(): the first of the other nodes is entered and updated more than
    // once where that lets warps begin with the rows of a core whose inner
    // columns are whole warps: shared-memory wavefronts of 900 x 300, 66 x 30 nodes a
    // CTA, 5.0 -> 3.5 k a step, 4.2 -> 3.9 us in the total-energy mode; 700 x 200
    // 2.9 -> 2.4)
    const int n_core = w * h, n_edge = res_edges(R, t), n_nodes = res_nodes(t, R.depth - 1);
    const int fill = fills<S, TM>() ? res_fill(R, t) : 0, n_items = n_nodes + fill;
    for (int e = tid; e < n_items; e += T) {
        const int q = e < n_edge ? e : max(e - fill, n_edge);
        int c, r;
        if (q < n_core)
            res_core_node(R, t, q, &c, &r);
        else
            res_shell_node(t, q - n_core, &c, &r);
        item[e] = (unsigned)(origin + r * RS + c) | (q < n_edge ? res_cell(R, t, c, r) : kNoCell) << 16 |
                  (wraps && r == h - 1 ? kWrapUp : 0u) | (wraps && r == 0 ? kWrapDown : 0u);
    }
    const int n_halo = R.cells > 0 ? res_nodes(t, R.depth) - n_core : 0;
    for (int q = tid; q < n_halo; q += T) {
        int c, r;
        res_shell_node(t, q, &c, &r);
        unsigned cell;
        const int from = res_owner(R, G.nx, G.ny, perx, pery, t, c, r, &cell);
        halo_src[q] = (unsigned)(from * R.cells) + cell;
        halo_dst[q] = (unsigned short)(origin + r * RS + c);
    }
    const ResGhosts ghosts = res_ghosts(R, G.nx, G.ny, perx, pery, t);
    const int n_ghost = ghosts.w + ghosts.e + ghosts.s + ghosts.n;
    for (int q = tid; q < n_ghost; q += T) {
        const ResGhost g = res_ghost(ghosts, G.nx, G.ny, perx, pery, t, q);
        const int dst = origin + g.r * RS + g.c, src = origin + g.sr * RS + g.sc;
        ghost[q] = make_uint2((unsigned)dst | (unsigned)src << 16, (unsigned)g.side | (unsigned)g.along << 2);
    }
    if (tid < R.depth) upto[tid] = res_nodes(t, tid) + fill;
    if (tid < 4) split_now[0][tid] = split_at(G, tid, A.level0 + 1);
    // the tile, ghost cells of the level included
    {
        const int c0 = -min(t.l + 1, pad_x), c1 = min(w + t.r, w + pad_x - 1);
        const int r0 = -min(t.b + 1, pad_y), r1 = min(h + t.t, h + pad_y - 1);
        const int cols = c1 - c0 + 1, per = 9 * cols, n = (r1 - r0 + 1) * per;
        for (int q = tid; q < n; q += T) {
            const int j = q / per, k = q - j * per, i = k / cols, c = c0 + k - i * cols, r = r0 + j;
            int gx = x0 + c, gy = y0 + r;
            if (R.px > 1 && perx) gx = (gx + G.nx * R.depth) % G.nx;
            if (R.py > 1 && pery) gy = (gy + G.ny * R.depth) % G.ny;
            cur[origin + r * RS + i * P + c] =
                A.fin[(size_t)(gy + 1) * (size_t)G.row + i * pl + (size_t)(gx + PADX)];
        }
    }
    __syncthreads();

    constexpr int Q = kCellWords<S>;
    const size_t slot_cells = (size_t)gridDim.x * R.cells;
    // the last warps poll, those before them fill ghost cells; FP32: after the
    // very last one, which follows the moving splits, beside the node updates
    // (its few FP64 instructions take up to 1600 cycles)
    const int T1 = sizeof(S) == 4 ? T - 32 : T;
    const int halo_tid = tid < T1 ? T1 - 1 - tid : tid;
    const int ghost_tid = (halo_tid - (n_halo + 31) / 32 * 32 % T + T) % T;
    const int split_tid = sizeof(S) == 4 ? tid - T1 : tid;
    unsigned bits = 0;
    bool ok = true;
    // j: the step's place since the last exchange, round: exchanges so far
    for (int s = 0, j = R.depth - A.first, round = 0; s < A.nsteps; ++s) {
        const unsigned tag = epoch + (unsigned)round + 1u;
        const bool more = s + 1 < A.nsteps, keep = s >= A.write_from;
        const bool publish = more && j == R.depth - 1;
        // steps from here to the next exchange, or to the end, this one included
        const int n_now = upto[min(R.depth - j, A.nsteps - s) - 1];
        const ResWord* in_box = A.xch + (tag & 1u) * slot_cells * Q;
        ResWord* out_box = publish ? A.xch + ((tag & 1u) * slot_cells + (size_t)cta * R.cells) * Q : nullptr;
        if (more && split_tid >= 0 && split_tid < 4)
            split_now[(s + 1) & 1][split_tid] = split_at(G, split_tid, A.level0 + s + 2);
        if constexpr (sizeof(S) == 8) {
            bits |= quad_update(M, cur, nxt, item, n_now, P, around);
            __syncthreads();  // a node's values come from four warps
            for (int q = tid; q < n_edge && publish; q += T) {
                const unsigned it = item[q];
                ResWord* d = out_box + (size_t)item_cell(it) * Q;
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const double v = nxt[item_place(it) + i * P];
                    st_word(d + i, (unsigned)__double2loint(v), (unsigned)__double2hiint(v), 0u, tag);
                }
            }
        } else {
            for (int q = tid < T1 ? tid : n_now; q < n_now; q += T1) {
                const unsigned it = item[q];
                const int at = item_place(it);
                S o[9];
                bits |= node_update<TM>(M, cur + at, P, it & kWrapUp ? -around : RS, it & kWrapDown ? around : -RS, o);
#pragma unroll
                for (int i = 0; i < 9; ++i) nxt[at + i * P] = o[i];
                if (publish && item_cell(it) != kNoCell) {
                    ResWord* d = out_box + (size_t)item_cell(it) * Q;
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        st_word(d + k, __float_as_uint(o[3 * k]), __float_as_uint(o[3 * k + 1]),
                                __float_as_uint(o[3 * k + 2]), tag);
                }
            }
        }
        if (sizeof(S) == 4 && (keep || n_ghost)) __syncthreads();
        if (keep) {
            // this level goes to the context's buffer too
            S* const fout = ((s & 1) ? A.out_odd : A.out_even) + (size_t)(s >> 1) * (size_t)A.out_stride;
            const int cols = 9 * w;
            for (int q = tid; q < h * cols; q += T) {
                const int r = q / cols, k = q - r * cols, i = k / w, c = k - i * w;
                fout[cell(G, x0 + c, y0 + r) + i * pl] = nxt[origin + r * RS + i * P + c];
            }
            for (int q = tid; q < 2 * (w + h); q += T) {
                const int k = q < 2 * w ? q >> 1 : (q - 2 * w) >> 1;
                const int c = q < 2 * w ? k : (q & 1 ? w - 1 : 0), r = q < 2 * w ? (q & 1 ? h - 1 : 0) : k;
                const int ix = x0 + c, iy = y0 + r;
                if (ix == 0 || iy == 0 || ix == G.nx - 1 || iy == G.ny - 1) {
                    S v[9];
#pragma unroll
                    for (int i = 0; i < 9; ++i) v[i] = nxt[origin + r * RS + i * P + c];
                    write_ghosts(G, fout, ix, iy, v, A.level0 + s + 1);
                }
            }
        }
        if (!more) break;
        for (int q = halo_tid; q < n_halo && ok && publish; q += T)
            ok = receive<S>(in_box + (size_t)halo_src[q] * Q, tag, nxt + halo_dst[q], P, A.status);
        // (ghost cells beside the shells are made from received cells)
        if (publish && n_ghost && R.depth > 1) __syncthreads();
        for (int q = ghost_tid; q < n_ghost; q += T) {
            const uint2 e = ghost[q];
            const int side = e.y & 3u;
            fill_ghost(G, side, (int)(e.y >> 2) < split_now[s & 1][side] ? 0 : 1, nxt + (e.x & 0xffffu),
                       nxt + (e.x >> 16), P);
        }
        if (__syncthreads_or(!ok)) {
            ok = false;
            break;
        }
        S* swap = cur;
        cur = nxt;
        nxt = swap;
        j = publish ? 0 : j + 1;
        round += publish;
    }
    if (!ok) bits |= ST_TIMEOUT;
    report(A.status, bits);
    // every CTA has read the tag counter before it counts itself out
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(A.sync + 1, 1u) == gridDim.x - 1) {
            A.sync[0] = epoch + (unsigned)A.nsteps;
            A.sync[1] = 0u;
            __threadfence();
        }
    }
}

namespace {
constexpr int kThreads32 = 768, kThreads64 = 128 * kQuadGroups;

// The largest dynamic shared memory of a plan: 227 KB a CTA less the static
// part; FP64 tiles are small.
template <typename S>
constexpr size_t kSmemMax = sizeof(S) == 4 ? 226 * 1024 : 113 * 1024;

size_t smem_bytes(const ResPlan& R, size_t esize) {
    const ResTile full = res_full_tile(R);
    return 2 * (size_t)(R.bh + 2 * res_pad_y(R)) * 9 * R.pitch * esize + 8 * (size_t)res_max_ghosts(R) +
           6 * (size_t)(res_nodes(full, R.depth) - R.bw * R.bh) + 4 * (size_t)(res_nodes(full, R.depth - 1) + kMaxFill);
}

template <typename S, int TM>
constexpr auto kernel_of() {
    if constexpr (sizeof(S) == 4)
        return k_resident<float, TM, kThreads32, Model<float>>;
    else
        return k_resident<double, TM, kThreads64, Fp64Step>;
}
}  // namespace

// The split of a grid over at most one CTA per SM: for every number of tiles
// in y the fewest columns that fit, as they are, rounded up to 32 (a warp's
// nodes then lie in one row) or to whole warps; the cheapest by an estimate of
// the step's time in us, fitted to 260 splits of grids from 400 x 4 to 1240 x
// 310 (7 % rms): per warp of nodes, per cell exchanged, for neighbours in y,
// and per CTA (the more, the more often one lags).  Tiles that span the grid's
// height exchange every depth-th step, at 0.4 us (0.7 in FP64) an exchange
// besides: one to four steps, 2000 x 4 1.35 / 1.11 / 1.02 / 0.99 us a step, FP64
// 400 x 4 3.05 / 2.67 / 2.60 / 3.25 (the fourth takes another 32 nodes); six
// and eight gain nothing more.  With neighbours on both axes deeper tiles gain
// at most 6 % (128 x 32) and lose from 512 x 128 on.  FP64: only up to kQuadGroups groups of 32
// nodes per SM (beyond, a launch a step keeps the FP64 pipe as busy: 400 x 100
// 11.1 us a step, 12.6 in a resident kernel of one node a thread).
template <typename S, int TM>
bool resident_plan(int nx, int ny, ResPlan* best) {
    constexpr bool f64 = sizeof(S) == 8;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) {
        cudaGetLastError();
        return false;
    }
    if ((long long)nx * ny > (long long)sms * (f64 ? 32 * kQuadGroups : 3000)) return false;
    double cost = 0.0;
    bool found = false;
    for (int py = 1; py <= ny && py <= sms; ++py)
        for (int how = 0; how < 3; ++how) {
            ResPlan R{};
            R.bh = (ny + py - 1) / py;
            R.py = (ny + R.bh - 1) / R.bh;
            if (R.py != py) continue;
            const int mx = sms / py;
            R.bw = (nx + mx - 1) / mx;
            const int ends = R.bw < nx ? 2 : 0;  // columns updated apart from the rows
            if (how == 1) R.bw = (R.bw - ends + 31) / 32 * 32 + ends;
            if (how == 2 && R.bh < 32) R.bw = (R.bw + 32 / R.bh - 1) / (32 / R.bh) * (32 / R.bh);
            R.px = (nx + R.bw - 1) / R.bw;
            for (R.depth = 1; R.depth <= (R.py == 1 && R.px > 1 ? kMaxDepth : 1); ++R.depth) {
                // pitch: a warp that continues on the next row of the inner
                // columns stays free of bank conflicts if 9 pitch = their
                // number modulo 32 banks (9 x 25 = 1 mod 32); if rows are whole
                // warps, an odd pitch keeps the column updates free of them
                const int inner = R.bw - (R.px > 1 ? min(2 * R.depth, R.bw) : 0);
                R.pitch = R.bw + 2 * res_pad_x(R);
                if (inner % 32 != 0)
                    R.pitch += ((25 * inner - R.pitch) % 32 + 32) % 32;
                else
                    R.pitch |= 1;
                R.cells = res_cells(R);
                const ResTile full = res_full_tile(R);
                const int warps = (res_nodes(full, R.depth - 1) + (fills<S, TM>() ? res_fill(R, full) : 0) + 31) / 32;
                const int received = res_nodes(full, R.depth) - R.bw * R.bh;
                if (f64) {
                    if (warps > kQuadGroups) continue;
                    R.threads = 128 * warps;
                } else {
                    const int most = kThreads32 - 32, rounds = (32 * warps + most - 1) / most;
                    R.threads = (warps + rounds - 1) / rounds * 32;
                    // warps enough to poll beside those that update the last nodes
                    const int roles = (received + 31) / 32 * 32 + 64;
                    if (R.threads < roles) R.threads = roles < most ? roles : most;
                    R.threads += 32;
                }
                R.smem = smem_bytes(R, sizeof(S));
                // places in the tile are 16-bit, and cells but for one value
                if ((R.bh + 2 * res_pad_y(R)) * 9 * R.pitch > 65535 || R.cells >= (int)kNoCell ||
                    R.smem > kSmemMax<S>)
                    continue;
                double sum = 0.0;  // warps of nodes over the steps to an exchange
                for (int d = 0; d < R.depth; ++d) sum += f64 ? warps : (res_nodes(full, d) + 31) / 32;
                const double each = f64 ? 1.25 : TM == T_INT64 ? 0.13 : inner % 32 == 0 ? 0.060 : 0.067;
                const double c = (each * sum + (f64 ? 0.02 : 0.002) * received + (R.py > 1 ? 0.2 : 0.0) +
                                  (f64 ? 0.7 : 0.4)) / R.depth + 0.001 * R.px * R.py;
                if (!found || c < cost) {
                    found = true;
                    cost = c;
                    *best = R;
                }
            }
        }
    if (!found) return false;
    best->xch_bytes = 2 * (size_t)best->px * best->py * best->cells * kCellWords<S> * sizeof(ResWord);
    // one CTA per SM is always resident: the launch bounds and kSmemMax see to
    // it (a device with fewer SMs free refuses the cooperative launch)
    if (allow_smem<kernel_of<S, TM>()>(kSmemMax<S>) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return true;
}

// A launch costs 10 to 40 us besides its steps, the more the larger the tiles
// (their level read, the last two written), and a step in it saves what the
// tile kernel's launch and drain take, 2 to 4 us, or with the FP64 sum and on
// thin FP64 grids 2 to 5.  Where the two meet, in steps, and per node of a tile
// the line above it taken here (us a call, launches of a step / one launch):
// FP32_CONS 400 x 4 (12 nodes) 4, 400 x 100 (280) 6, 512 x 256 (900) 8, 900 x 300
// (1950) 11 (n = 8: 53 / 61, 24: 159 / 119), 1240 x 310 (2574) 13 (n = 8: 62 /
// 74, 24: 184 / 150); FP32_TDF 4, 6, 9, 15, 13; FP32_T64 4, 5, 5, 6, 10.  With
// every level written a step also stores a level, as the tile kernel does, but
// with nothing to hide it: recomputation of 23 levels and their adjoint, 400 x
// 100 220 / 206, 512 x 128 (450) 239 / 235, 512 x 256 325 / 340, 900 x 300 414 /
// 512 (FP32_T64 274 / 246, 296 / 286, 439 / 423, 598 / 634).  FP64, where a step
// by launches takes 6.0 us: one group of 32 nodes a CTA 4 steps, two groups 5 to
// 30 with their number of nodes (64: 5.8 us a step), three 10 on thin grids (4.9
// to 5.2) and none on others (7.2); with every level written two groups win from
// the start (a launch less on the host beside the adjoint's) and three lose.
template <typename S, int TM>
int resident_min_steps(const ResPlan& R, bool all_levels) {
    const int nodes = R.bw * R.bh;
    int n;
    if (sizeof(S) == 8) {
        const int groups = (nodes + 31) / 32;
        if (all_levels)
            n = groups <= 2 ? kResidentFewest : INT_MAX;
        else if (groups == 1)
            n = 4;
        else if (R.py == 1)
            n = groups == 2 ? 5 : 10;
        else
            n = groups == 2 ? 5 + (nodes - 32) * (nodes - 32) / 40 : INT_MAX;
    } else if (TM == T_INT64) {
        n = !all_levels ? 5 + nodes / 400 : nodes <= 950 ? 5 + nodes / 60 : INT_MAX;
    } else {
        n = !all_levels ? 6 + nodes / 220 : nodes <= 320 ? 7 + nodes / 50 : INT_MAX;
    }
    return n;
}

// A stalled launch leaves its last CTA out, which makes the halves of the
// exchange buffer smaller by its cells.  The cells that the others then wait
// for still lie in the buffer: behind their half, where there are tags of the
// other parity, or of earlier launches.
template <typename S, int TM>
cudaError_t launch_resident(const ResPlan& R, const Model<S>& M, const Fp64Step& M64, const Grid<S>& G,
                            const ResRun<S>& A, bool stall, cudaStream_t st) {
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3(R.px * R.py - (stall ? 1 : 0));
    lc.blockDim = dim3(R.threads);
    lc.dynamicSmemBytes = R.smem;
    lc.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    if constexpr (sizeof(S) == 4)
        return cudaLaunchKernelEx(&lc, kernel_of<S, TM>(), M, G, R, A);
    else
        return cudaLaunchKernelEx(&lc, kernel_of<S, TM>(), M64, G, R, A);
}

cudaError_t resident_set_wait_cycles(long long cycles) {
    return cudaMemcpyToSymbol(g_poll_cycles, &cycles, sizeof(cycles));
}

#define LBM_RES_INST(S, TM)                                                                              \
    template bool resident_plan<S, TM>(int, int, ResPlan*);                                              \
    template int resident_min_steps<S, TM>(const ResPlan&, bool);                                        \
    template cudaError_t launch_resident<S, TM>(const ResPlan&, const Model<S>&, const Fp64Step&,        \
                                                const Grid<S>&, const ResRun<S>&, bool, cudaStream_t);
LBM_RES_INST(double, T_PLAIN)
LBM_RES_INST(float, T_INT32)
LBM_RES_INST(float, T_INT64)
LBM_RES_INST(float, T_DF)
LBM_RES_INST(float, T_CONS)
#undef LBM_RES_INST

}  // namespace lbm
