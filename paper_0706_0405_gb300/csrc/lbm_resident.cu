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
// 5.3 -> 1.2 / 3.6 -> 1.2 / 4.5 -> 1.5, 2000 x 4 5.4 -> 1.3 / 3.7 -> 1.2 /
// 4.5 -> 1.6, 400 x 100 6.1 -> 2.0 / 4.7 -> 1.8 / 5.8 -> 2.5, 1024 x 256
// 8.8 -> 5.4 / 7.3 -> 4.5 / 11.4 -> 7.0; FP64: 400 x 4 6.1 -> 2.9,
// 2000 x 4 6.0 -> 3.9.  A small tile's step is a chain of latencies: the node
// update 750 cycles, the exchange about 1000, barriers; a large one's is
// issue- and shared-memory-bound (41 % of the issue slots at 1024 x 256, the
// exchange not overlapped).
//  * two copies of the tile with a one-cell halo, [row][population][column]
//    like a level; a step reads one and writes the other;
//  * a step is: every thread updates its nodes; a CTA barrier; then different
//    warps publish the tile's edge cells, fill its ghost cells and poll its
//    halo cells, one cell (nine values) a thread, from tables made at the
//    start (source and target of every cell); a second barrier.  (In the edge
//    nodes' own threads this took up to 3600 cycles a step, where the node
//    update takes 750; one value a thread was slower too, its polls one after
//    the other);
//  * an edge value travels as one 64-bit word, the value and the step it
//    belongs to (FP64: two words, a half of the value each), written and
//    polled with relaxed GPU-scope accesses.  The tag makes the word its own
//    flag: no fence, no second round trip (500 cycles one way, measured
//    between two CTAs).  Slots alternate by the step's parity: a CTA publishes
//    step t + 2 only after it has received its neighbours' t + 1, which they
//    publish after a barrier that follows their reads of t.  Tags come from a
//    counter in device memory that only grows, advanced by the last CTA to
//    leave, so replays of a captured launch work;
//  * the place of a moving split (the double Mach reflection's top boundary)
//    is turned into an index once a step, by the last warp;
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

__device__ __forceinline__ void st_word(unsigned long long* p, unsigned value, unsigned tag) {
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(((unsigned long long)tag << 32) | value) : "memory");
}
__device__ __forceinline__ unsigned long long ld_word(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Words per value, and the value's transport.
template <typename S>
constexpr int kWords = sizeof(S) / 4;
__device__ __forceinline__ void put(unsigned long long* p, float v, unsigned tag) {
    st_word(p, __float_as_uint(v), tag);
}
__device__ __forceinline__ void put(unsigned long long* p, double v, unsigned tag) {
    st_word(p, (unsigned)__double2loint(v), tag);
    st_word(p + 1, (unsigned)__double2hiint(v), tag);
}
__device__ __forceinline__ float take(const unsigned long long (&w)[1]) { return __uint_as_float((unsigned)w[0]); }
__device__ __forceinline__ double take(const unsigned long long (&w)[2]) {
    return __hiloint2double((int)(unsigned)w[1], (int)(unsigned)w[0]);
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
                                                const unsigned short* item, int n_items, int P) {
    __shared__ double pairs[kQuadGroups][8][32];  // differences (0..3) and sums (4..7) of the warps' pairs
    __shared__ double mom[kQuadGroups][5][32];    // 1 / rho, rho, gx, gy, E / b
    const int lane = threadIdx.x & 31, role = threadIdx.x / 32 & 3, group = threadIdx.x / 128;
    const int q = group * 32 + lane;
    const bool in = q < n_items;
    const int at = item[in ? q : 0];
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

// Poll the nine values of one halo cell until all carry the tag, and put them
// at dst (P apart).  False if the poll gave up.
template <typename S>
__device__ __forceinline__ bool receive(const unsigned long long* src, int stride, unsigned tag, S* dst, int P,
                                        const unsigned* status) {
    constexpr int W = kWords<S>;
    unsigned long long w[9][W];
    long long t0 = 0;
    for (unsigned spins = 0;; ++spins) {
#pragma unroll
        for (int i = 0; i < 9; ++i)
#pragma unroll
            for (int k = 0; k < W; ++k) w[i][k] = ld_word(src + (size_t)(i * stride + k));
        unsigned miss = 0;
#pragma unroll
        for (int i = 0; i < 9; ++i)
#pragma unroll
            for (int k = 0; k < W; ++k) miss |= (unsigned)(w[i][k] >> 32) ^ tag;
        if (miss == 0) break;
        if ((spins & 63) == 63) {
            const long long t = clock64();
            if (t0 == 0) t0 = t;
            if (t - t0 > kPollCycles || (*(volatile const unsigned*)status & ST_TIMEOUT)) return false;
        }
    }
#pragma unroll
    for (int i = 0; i < 9; ++i) dst[i * P] = take(w[i]);
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
    // index; per halo cell its source's word; per published cell its place and
    // its cell index; per halo cell its place; per node its place
    uint2* ghost = reinterpret_cast<uint2*>(nxt + buf);
    unsigned* halo_src = reinterpret_cast<unsigned*>(ghost + R.cells);
    unsigned* send = halo_src + R.cells;
    unsigned short* halo_dst = reinterpret_cast<unsigned short*>(send + R.cells);
    unsigned short* item = halo_dst + R.cells;
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

    const int n_items = w * h;  // the tile's nodes, row by row
    for (int q = tid; q < n_items; q += T) item[q] = (unsigned short)(origin + q / w * RS + q % w);
    // halo cells that come from other CTAs: west and east columns, south and
    // north rows.  A CTA's published cells: bottom row, top row (bw each),
    // left column, right column (bh each)
    const int n_w = west >= 0 ? h : 0, n_e = east >= 0 ? h : 0, n_s = south >= 0 ? w : 0, n_n = north >= 0 ? w : 0;
    const int n_halo = n_w + n_e + n_s + n_n;  // also the number of cells published
    const int cta_words = 9 * R.cells;
    for (int q = tid; q < n_halo; q += T) {
        int k = q, from, at, dst, src, to;
        if (k < n_w) {
            from = west, at = 2 * R.bw + R.bh + k, dst = origin + k * RS - 1;
            src = origin + k * RS, to = 2 * R.bw + k;
        } else if ((k -= n_w) < n_e) {
            from = east, at = 2 * R.bw + k, dst = origin + k * RS + w;
            src = dst - 1, to = 2 * R.bw + R.bh + k;
        } else if ((k -= n_e) < n_s) {
            from = south, at = R.bw + k, dst = origin - RS + k;
            src = origin + k, to = k;
        } else {
            k -= n_s;
            from = north, at = k, dst = origin + h * RS + k;
            src = dst - RS, to = R.bw + k;
        }
        halo_src[q] = (unsigned)(from * cta_words + at);
        halo_dst[q] = (unsigned short)dst;
        send[q] = (unsigned)src | (unsigned)to << 16;
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

    constexpr int W = kWords<S>;
    unsigned long long* const mine = A.xch + (size_t)cta * cta_words * W;
    const size_t slot_words = (size_t)gridDim.x * cta_words * W;
    // the first warps publish, the next fill ghost cells, the next poll
    const int ghost_from = (n_halo + 31) / 32 * 32 % T, halo_from = (ghost_from + (n_ghost + 31) / 32 * 32) % T;
    const int ghost_tid = (tid - ghost_from + T) % T, halo_tid = (tid - halo_from + T) % T;
    unsigned bits = 0;
    bool ok = true;
    for (int s = 0; s < A.nsteps; ++s) {
        const unsigned tag = epoch + (unsigned)s + 1u;
        if constexpr (sizeof(S) == 8) {
            bits |= quad_update(M, cur, nxt, item, n_items, P);
        } else {
            for (int q = tid; q < n_items; q += T) {
                const int at = item[q];
                S o[9];
                bits |= node_update<TM>(M, cur + at, P, o);
#pragma unroll
                for (int i = 0; i < 9; ++i) nxt[at + i * P] = o[i];
            }
        }
        __syncthreads();
        if (s >= A.write_from) {
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
        if (s + 1 == A.nsteps) break;
        unsigned long long* const out_box = mine + (tag & 1u) * slot_words;
        for (int q = tid; q < n_halo; q += T) {
            const unsigned e = send[q];
            const S* v = nxt + (e & 0xffffu);
            unsigned long long* d = out_box + (size_t)(e >> 16) * W;
#pragma unroll
            for (int i = 0; i < 9; ++i) put(d + (size_t)(i * R.cells * W), v[i * P], tag);
        }
        for (int q = ghost_tid; q < n_ghost; q += T) {
            const uint2 e = ghost[q];
            const int side = e.y & 3u;
            fill_ghost(G, side, (int)(e.y >> 2) < split_now[s & 1][side] ? 0 : 1, nxt + (e.x & 0xffffu),
                       nxt + (e.x >> 16), P);
        }
        const unsigned long long* in_box = A.xch + (tag & 1u) * slot_words;
        for (int q = halo_tid; q < n_halo && ok; q += T)
            ok = receive<S>(in_box + (size_t)halo_src[q] * W, R.cells * W, tag, nxt + halo_dst[q], P, A.status);
        if (tid >= T - 4) split_now[(s + 1) & 1][T - 1 - tid] = split_at(G, T - 1 - tid, A.level0 + s + 2);
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
constexpr int kThreads32 = 512, kThreads64 = 128 * kQuadGroups;

// The largest dynamic shared memory of a plan: 227 KB a CTA less the static
// part; FP64 tiles are small.
template <typename S>
constexpr size_t kSmemMax = sizeof(S) == 4 ? 226 * 1024 : 113 * 1024;

size_t smem_bytes(const ResPlan& R, size_t esize) {
    return 2 * (size_t)(R.bh + 2) * 9 * R.pitch * esize + 18 * (size_t)R.cells + 2 * (size_t)R.bw * R.bh;
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
            const int align = how == 0 ? 1 : how == 1 ? 32 : R.bh < 32 ? 32 / R.bh : 1;
            const int mx = sms / py;
            R.bw = ((nx + mx - 1) / mx + align - 1) / align * align;
            R.px = (nx + R.bw - 1) / R.bw;
            // pitch: a warp that continues on the next row stays free of bank
            // conflicts if 9 pitch = bw modulo 32 banks (9 x 25 = 1 mod 32)
            R.pitch = R.bw + 4;
            if (R.bw % 32 != 0) R.pitch += ((25 * R.bw - R.pitch) % 32 + 32) % 32;
            R.cells = 2 * R.bw + 2 * R.bh;
            const int warps = (R.bw * R.bh + 31) / 32;
            const int exchanged = R.py > 1 ? R.cells : 2 * R.bh;
            if (f64) {
                if (warps > kQuadGroups) continue;
                R.threads = 128 * warps;
            } else {
                const int rounds = (32 * warps + kThreads32 - 1) / kThreads32;
                R.threads = (warps + rounds - 1) / rounds * 32;
                // warps enough that no warp has to publish and poll as well
                const int roles = 2 * ((exchanged + 31) / 32 * 32) + 64;
                if (R.threads < roles) R.threads = roles < kThreads32 ? roles : kThreads32;
            }
            R.smem = smem_bytes(R, sizeof(S));
            // places in the tile are 16-bit
            if ((R.bh + 2) * 9 * R.pitch > 65535 || R.smem > kSmemMax<S>) continue;
            const double each = f64 ? 1.25 : TM == T_INT64 ? 0.13 : R.bw % 32 == 0 ? 0.060 : 0.067;
            const double c = each * warps + 0.002 * exchanged + (R.py > 1 ? 0.2 : 0.0) + 0.001 * R.px * R.py;
            if (!found || c < cost) {
                found = true;
                cost = c;
                *best = R;
            }
        }
    if (!found) return false;
    best->xch_bytes = 2 * (size_t)best->px * best->py * 9 * best->cells * 8 * (sizeof(S) / 4);
    // resident all at once; sets the kernel's shared-memory limit on this device
    constexpr auto kern = kernel_of<S, TM>();
    int per_sm = 0;
    if (allow_smem<kernel_of<S, TM>()>(kSmemMax<S>) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, best->threads, best->smem) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return best->px * best->py <= per_sm * sms;
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
