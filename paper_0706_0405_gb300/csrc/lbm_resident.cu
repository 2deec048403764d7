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
// 5.3 -> 1.3 / 3.6 -> 1.2 / 4.5 -> 1.6, 2000 x 4 5.4 -> 1.3 / 3.7 -> 1.2 /
// 4.5 -> 1.6, 400 x 100 6.1 -> 1.9 / 4.7 -> 1.7 / 5.8 -> 2.4, 1024 x 256
// 8.8 -> 4.5 / 7.3 -> 3.8 / 11.4 -> 6.8; FP64: 400 x 4 6.1 -> 3.1,
// 2000 x 4 6.0 -> 4.0.  A small tile's step is a chain of latencies: the node
// update 950 cycles, the exchange about 1300 (of which 1000 from one CTA's
// store to another's poll, measured between neighbours among 50 to 125 CTAs),
// barriers 150; a large one's is issue- and shared-memory-bound.
//  * two copies of the tile with a one-cell halo, [row][population][column]
//    like a level; a step reads one and writes the other;
//  * a step is: the threads update the tile's nodes, its edge nodes first,
//    and publish the edge nodes' values from registers as they go; the
//    last warps poll the halo cells, one cell (nine values) a thread, while
//    others fill the tile's ghost cells from tables made at the start; a
//    barrier ends the step, and one before the ghost cells where the tile has
//    any.  (Publishing in a phase of its own after a barrier cost 0.35 us a
//    step; ghost rules and polls in the edge nodes' own threads up to 3600
//    cycles, where the node update takes 900);
//  * edge values travel as 128-bit words of three 32-bit values and the step
//    they belong to (FP64: one value), written and polled with relaxed
//    GPU-scope accesses.  The tag makes a word its own flag: no fence, no
//    second round trip.  Slots
//    alternate by the step's parity: a CTA publishes step t + 2 only after it
//    has received its neighbours' t + 1, which they publish after a barrier
//    that follows their reads of t.  Tags come from a counter in device memory
//    that only grows, advanced by the last CTA to leave, so replays of a
//    captured launch work;
//  * the place of a moving split (the double Mach reflection's top boundary)
//    is turned into an index once a step, by a warp of its own;
//  * the last two steps also write their levels to the context's buffers,
//    ghosts included, so that every call leaves what the one-step kernels
//    would have left.
// Polls are bounded: on give-up the CTA raises ST_TIMEOUT and leaves, and so
// do the others, which watch that word while they poll.
#include "lbm_launch.h"

namespace lbm {

namespace {
constexpr long long kPollCycles = 4000000000LL;  // ~2 s, then a poll gives up
constexpr int kPadL = 2;                         // columns left of the tile in shared memory (pairs stay aligned)

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

constexpr unsigned kNoCell = 0xffffu;
// The exchange cell of node (lx, ly) of a tile of w x h nodes: the bottom
// row, the top row, the left and the right column, where there are CTAs on
// that axis.
__host__ __device__ __forceinline__ unsigned cell_id(const ResPlan& R, int lx, int ly, int w, int h) {
    if (R.py > 1) {
        if (ly == 0) return lx;
        if (ly == h - 1) return R.bw + lx;
    }
    if (R.px > 1) {
        if (lx == 0) return 2 * R.bw + ly;
        if (lx == w - 1) return 2 * R.bw + R.bh + ly;
    }
    return kNoCell;
}

// Values of one node after a step, FP32 modes, from the box b (populations P
// apart, rows 9 P).
template <int TM>
__device__ __forceinline__ unsigned node_update(const Model<float>& M, const float* b, int P, float (&o)[9]) {
    float f[9], rho, ux, uy, T;
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = b[i * P];
    moments<float, TM>(f, M, rho, ux, uy, T);
    relaxation<float, TM>(M, f, rho, ux, uy, T, o);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const float* p = b + i * P;
        o[i] = update(M, i, o[i], f[i], p[1], p[-1], p[9 * P], p[-9 * P]);
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
                                                const unsigned* item, int n_items, int P) {
    __shared__ double pairs[kQuadGroups][8][32];  // differences (0..3) and sums (4..7) of the warps' pairs
    __shared__ double mom[kQuadGroups][5][32];    // 1 / rho, rho, gx, gy, E / b
    const int lane = threadIdx.x & 31, role = threadIdx.x / 32 & 3, group = threadIdx.x / 128;
    const int q = group * 32 + lane;
    const bool in = q < n_items;
    const int at = (int)(item[in ? q : 0] & 0xffffu);
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
        nxt[at + i * P] = fp64_update(C, i, r, c, n[1], n[-1], n[9 * P], n[-9 * P]);
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
            if (t - t0 > kPollCycles || (*(volatile const unsigned*)status & ST_TIMEOUT)) return false;
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
    const int T = blockDim.x, tid = threadIdx.x;
    const int cta = blockIdx.x, bx = cta % R.px, by = cta / R.px;
    const int x0 = bx * R.bw, y0 = by * R.bh;
    const int w = min(R.bw, G.nx - x0), h = min(R.bh, G.ny - y0);
    const size_t buf = (size_t)(R.bh + 2) * RS;
    S* cur = reinterpret_cast<S*>(smem);
    S* nxt = cur + buf;
    // tables: per ghost cell its place, its source's, its side and along-side
    // index; per halo cell its source's cell; per node its place and the cell
    // it is published as; per halo cell its place
    uint2* ghost = reinterpret_cast<uint2*>(nxt + buf);
    unsigned* halo_src = reinterpret_cast<unsigned*>(ghost + R.cells);
    unsigned* item = halo_src + R.cells;
    unsigned short* halo_dst = reinterpret_cast<unsigned short*>(item + R.bw * R.bh);
    __shared__ int split_now[2][4];  // by the step's parity
    const int origin = RS + kPadL;  // node (0, 0), population 0, in a buffer
    const unsigned epoch = *(volatile unsigned*)A.sync;
    const size_t pl = (size_t)G.plane;

    // neighbours: CTA index, -1 at a physical side or where the tile meets itself
    const bool perx = G.kind_lo[S_LEFT] == BC_PERIODIC, pery = G.kind_lo[S_BOTTOM] == BC_PERIODIC;
    const int west = bx > 0 ? cta - 1 : (perx && R.px > 1 ? cta + R.px - 1 : -1);
    const int east = bx < R.px - 1 ? cta + 1 : (perx && R.px > 1 ? cta - (R.px - 1) : -1);
    const int south = by > 0 ? cta - R.px : (pery && R.py > 1 ? cta + (R.py - 1) * R.px : -1);
    const int north = by < R.py - 1 ? cta + R.px : (pery && R.py > 1 ? cta - (R.py - 1) * R.px : -1);

    // the tile's nodes in the order of their update: those that are published
    // first (bottom and top row, left and right column, on the axes with other
    // CTAs), so that few warps publish, then the rest row by row
    const int n_items = w * h;
    const int ey = R.py > 1, ex = R.px > 1;
    const int n_rows = ey ? w * min(h, 2) : 0, rest_h = ey ? max(h - 2, 0) : h;
    const int n_cols = ex ? rest_h * min(w, 2) : 0, rest_w = ex ? w - 2 : w;
    const int n_edge = n_rows + n_cols;
    for (int q = tid; q < n_items; q += T) {
        int r, c, k = q;
        if (k < n_rows) {
            r = k < w ? 0 : h - 1;
            c = k < w ? k : k - w;
        } else if ((k -= n_rows) < n_cols) {
            r = ey + k % rest_h;
            c = k < rest_h ? 0 : w - 1;
        } else {
            k -= n_cols;
            r = ey + k / rest_w;
            c = ex + k % rest_w;
        }
        item[q] = (unsigned)(origin + r * RS + c) | cell_id(R, c, r, w, h) << 16;
    }
    // halo cells that come from other CTAs: west and east columns, south and
    // north rows
    const int n_w = west >= 0 ? h : 0, n_e = east >= 0 ? h : 0, n_s = south >= 0 ? w : 0, n_n = north >= 0 ? w : 0;
    const int n_halo = n_w + n_e + n_s + n_n;
    for (int q = tid; q < n_halo; q += T) {
        int k = q, from, dst;
        const int side = k < n_w ? S_LEFT : (k -= n_w) < n_e ? S_RIGHT : (k -= n_e) < n_s ? S_BOTTOM : S_TOP;
        if (side == S_LEFT) {
            from = west, dst = origin + k * RS - 1;
        } else if (side == S_RIGHT) {
            from = east, dst = origin + k * RS + w;
        } else if (side == S_BOTTOM) {
            from = south, dst = origin - RS + k;
        } else {
            k -= n_s;
            from = north, dst = origin + h * RS + k;
        }
        // the node in the other CTA's tile
        const int fw = min(R.bw, G.nx - from % R.px * R.bw), fh = min(R.bh, G.ny - from / R.px * R.bh);
        const int lx = side == S_LEFT ? fw - 1 : side == S_RIGHT ? 0 : k;
        const int ly = side == S_BOTTOM ? fh - 1 : side == S_TOP ? 0 : k;
        halo_src[q] = (unsigned)(from * R.cells) + cell_id(R, lx, ly, fw, fh);
        halo_dst[q] = (unsigned short)dst;
    }
    // ghost cells inside the tile: of physical sides, and of periodic sides
    // whose two ends the tile holds
    const int g_w = x0 == 0 && west < 0 ? h : 0, g_e = x0 + w == G.nx && east < 0 ? h : 0;
    const int g_s = y0 == 0 && south < 0 ? w : 0, g_n = y0 + h == G.ny && north < 0 ? w : 0;
    const int n_ghost = g_w + g_e + g_s + g_n;
    for (int q = tid; q < n_ghost; q += T) {
        int k = q, side, dst, src, along;
        if (k < g_w) {
            side = S_LEFT, dst = origin + k * RS - 1, src = perx ? dst + w : dst + 1, along = y0 + k;
        } else if ((k -= g_w) < g_e) {
            side = S_RIGHT, dst = origin + k * RS + w, src = perx ? dst - w : dst - 1, along = y0 + k;
        } else if ((k -= g_e) < g_s) {
            side = S_BOTTOM, dst = origin - RS + k, src = pery ? dst + h * RS : dst + RS, along = x0 + k;
        } else {
            k -= g_s;
            side = S_TOP, dst = origin + h * RS + k, src = pery ? dst - h * RS : dst - RS, along = x0 + k;
        }
        ghost[q] = make_uint2((unsigned)dst | (unsigned)src << 16, (unsigned)side | (unsigned)along << 2);
    }
    if (tid < 4) split_now[0][tid] = split_at(G, tid, A.level0 + 1);
    // the tile and its halo, ghost cells of the level included
    {
        const int cols = w + 2, per = 9 * cols, n = (h + 2) * per;
        for (int q = tid; q < n; q += T) {
            const int r = q / per, k = q - r * per, i = k / cols, c = k - i * cols;
            cur[r * RS + i * P + (kPadL - 1) + c] =
                A.fin[(size_t)(y0 + r) * (size_t)G.row + i * pl + (size_t)(x0 + c + PADX - 1)];
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
    for (int s = 0; s < A.nsteps; ++s) {
        const unsigned tag = epoch + (unsigned)s + 1u;
        const bool more = s + 1 < A.nsteps, keep = s >= A.write_from;
        const ResWord* in_box = A.xch + (tag & 1u) * slot_cells * Q;
        ResWord* out_box = more ? A.xch + ((tag & 1u) * slot_cells + (size_t)cta * R.cells) * Q : nullptr;
        if (more && split_tid >= 0 && split_tid < 4)
            split_now[(s + 1) & 1][split_tid] = split_at(G, split_tid, A.level0 + s + 2);
        if constexpr (sizeof(S) == 8) {
            bits |= quad_update(M, cur, nxt, item, n_items, P);
            __syncthreads();  // a node's values come from four warps
            for (int q = tid; q < n_edge && more; q += T) {
                const unsigned it = item[q];
                ResWord* d = out_box + (size_t)(it >> 16) * Q;
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const double v = nxt[(it & 0xffffu) + i * P];
                    st_word(d + i, (unsigned)__double2loint(v), (unsigned)__double2hiint(v), 0u, tag);
                }
            }
        } else {
            for (int q = tid < T1 ? tid : n_items; q < n_items; q += T1) {
                const unsigned it = item[q];
                const int at = (int)(it & 0xffffu);
                S o[9];
                bits |= node_update<TM>(M, cur + at, P, o);
#pragma unroll
                for (int i = 0; i < 9; ++i) nxt[at + i * P] = o[i];
                if (more && it >> 16 != kNoCell) {
                    ResWord* d = out_box + (size_t)(it >> 16) * Q;
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
        for (int q = halo_tid; q < n_halo && ok; q += T)
            ok = receive<S>(in_box + (size_t)halo_src[q] * Q, tag, nxt + halo_dst[q], P, A.status);
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
        S* t = cur;
        cur = nxt;
        nxt = t;
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
    return 2 * (size_t)(R.bh + 2) * 9 * R.pitch * esize + 14 * (size_t)R.cells + 4 * (size_t)R.bw * R.bh;
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
// nodes then lie in one row) or to whole warps; the cheapest by an estimate of the step's time
// in us, fitted to 260 splits of grids from 400 x 4 to 1240 x 310 (7 % rms):
// per warp of nodes, per cell exchanged, for neighbours in y, and per CTA (the
// more, the more often one lags).  FP64: only up to kQuadGroups groups of 32
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
            // pitch: a warp that continues on the next row of the inner columns
            // stays free of bank conflicts if 9 pitch = their number modulo 32
            // banks (9 x 25 = 1 mod 32); if rows are whole warps, an odd pitch
            // keeps the column updates free of them
            const int inner = R.bw - (R.px > 1 ? 2 : 0);
            R.pitch = R.bw + 4;
            if (inner % 32 != 0)
                R.pitch += ((25 * inner - R.pitch) % 32 + 32) % 32;
            else
                R.pitch |= 1;
            R.cells = 2 * R.bw + 2 * R.bh;
            const int warps = (R.bw * R.bh + 31) / 32;
            const int exchanged = R.py > 1 ? R.cells : 2 * R.bh;
            if (f64) {
                if (warps > kQuadGroups) continue;
                R.threads = 128 * warps;
            } else {
                const int most = kThreads32 - 32, rounds = (32 * warps + most - 1) / most;
                R.threads = (warps + rounds - 1) / rounds * 32;
                // warps enough to poll beside those that update the last nodes
                const int roles = (exchanged + 31) / 32 * 32 + 64;
                if (R.threads < roles) R.threads = roles < most ? roles : most;
                R.threads += 32;
            }
            R.smem = smem_bytes(R, sizeof(S));
            // places in the tile are 16-bit
            if ((R.bh + 2) * 9 * R.pitch > 65535 || R.smem > kSmemMax<S>) continue;
            const double each = f64 ? 1.25 : TM == T_INT64 ? 0.13 : inner % 32 == 0 ? 0.060 : 0.067;
            const double c = each * warps + (f64 ? 0.02 : 0.002) * exchanged + (R.py > 1 ? 0.2 : 0.0) + 0.001 * R.px * R.py;
            if (!found || c < cost) {
                found = true;
                cost = c;
                *best = R;
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

template <typename S, int TM>
cudaError_t launch_resident(const ResPlan& R, const Model<S>& M, const Fp64Step& M64, const Grid<S>& G,
                            const ResRun<S>& A, cudaStream_t st) {
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3(R.px * R.py);
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

#define LBM_RES_INST(S, TM)                                                                              \
    template bool resident_plan<S, TM>(int, int, ResPlan*);                                              \
    template cudaError_t launch_resident<S, TM>(const ResPlan&, const Model<S>&, const Fp64Step&,        \
                                                const Grid<S>&, const ResRun<S>&, cudaStream_t);
LBM_RES_INST(double, T_PLAIN)
LBM_RES_INST(float, T_INT32)
LBM_RES_INST(float, T_INT64)
LBM_RES_INST(float, T_DF)
LBM_RES_INST(float, T_CONS)
#undef LBM_RES_INST

}  // namespace lbm
