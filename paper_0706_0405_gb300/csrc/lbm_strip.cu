// lbm_strip.cu -- temporal blocking of a batch of thin problems (two or four
// rows, periodic in y, not periodic in x): one cooperative launch for all
// steps.  Each thread holds one column of a problem, all rows and populations
// of it in registers, so the y neighbours are the thread's own registers and
// the x neighbours come from the adjacent lanes by shuffles; no level is read
// from memory but at the start of a pass of up to 7 steps.
//
// The rows are updated two at a time in packed FP32x2 arithmetic, with every
// constant in shared memory in both lanes, ready to be an operand: 298 warp
// instructions per 32 nodes in the double-float mode, the columns computed
// twice included, where the tile kernel (one tensor copy per tile and step)
// issues 414.  Bound by the FP32 pipe's register reads: a packed FMA of three
// different operands takes three cycles on a quarter of an SM, two with one
// that the instruction before used too (measured), so that two, three and four
// warps to a scheduler take 24.6, 22.0 and 21.1 us a step on 256 tubes, and a
// fifth, with 96 registers a thread, 24.6.  In the 128 registers of four, the
// kernel of four rows spills 44 bytes a thread in the double-float mode, 20 in
// the total-energy mode and 232 with the FP64 sum.  Four CTAs of four warps
// to an SM, so that some load or store their columns while others compute: two
// of eight and one of sixteen take 3 and 5 % longer.  Against the tile kernel,
// us a step: 256 Riemann tubes 21.1 / 24.9 (total-energy mode 17.1 / 22.8), 64
// tubes 6.7 / 8.8, 4 tubes 1.9 / 4.0; with the FP64 sum of the temperature it
// is slower from 16 tubes on (40.6 / 34.9 us on 256), so the launch shape is
// left to lbm_batch_autotune.
#include "lbm_batch_plan.h"
#include "lbm_gridsync.cuh"
#include "lbm_launch.h"

namespace lbm {

namespace {
constexpr int kStripThreads = 32 * kStripWarps;
constexpr int kModelWords = sizeof(Model<float>) / sizeof(float);
static_assert(sizeof(Model<F2>) == 2 * sizeof(Model<float>), "the pair model is the model, word by word");

__device__ __forceinline__ F2 shfl_up(F2 a) { return F2{__shfl_up_sync(0xffffffffu, a.v, 1)}; }
__device__ __forceinline__ F2 shfl_down(F2 a) { return F2{__shfl_down_sync(0xffffffffu, a.v, 1)}; }

// One column on its way between threads: [population][row pair].
template <int NP>
struct __align__(16) Column {
    F2 f[9][NP];
    __device__ __forceinline__ void put(const F2 (&v)[9][NP]) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            if constexpr (NP == 2)
                *reinterpret_cast<ulonglong2*>(&f[i][0]) = make_ulonglong2(v[i][0].v, v[i][1].v);
            else
                f[i][0] = v[i][0];
        }
    }
    // population i, or with mirror the one that a wall across x reflects into it
    __device__ __forceinline__ void get(F2 (&v)[9][NP], bool mirror = false) const {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const F2* p = f[mirror ? mirror_x(i) : i];
            if constexpr (NP == 2) {
                const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(p);
                v[i][0].v = q.x;
                v[i][1].v = q.y;
            } else {
                v[i][0] = p[0];
            }
        }
    }
};

// The rule of a left or right side with `rows` rows if it is the same for all
// rows and times, and -1 otherwise.
__device__ __forceinline__ int side_rule(const Grid<float>& G, int side, int rows) {
    if (G.split_moving[side]) return -1;
    const int at = G.split_index[side];
    const int kind = at > 0 ? G.kind_lo[side] : G.kind_hi[side];
    return at <= 0 || at >= rows || (kind == G.kind_hi[side] && kind != BC_DIRICHLET) ? kind : -1;
}

// The ghost column on `side` of the level `level`, from the column beside it,
// where the side changes its rule along the rows or with time.
template <int NP>
__device__ __noinline__ void split_ghost(const Grid<float>& G, int side, const Column<NP>& src, long long level,
                                         Column<NP>& out) {
    for (int r = 0; r < 2 * NP; ++r) {
        const int part = side_part(G, side, r, level);
        const int kind = part ? G.kind_hi[side] : G.kind_lo[side];
        for (int i = 0; i < 9; ++i) {
            const float* s = reinterpret_cast<const float*>(src.f[kind == BC_REFLECT ? mirror_x(i) : i]);
            reinterpret_cast<float*>(out.f[i])[r] = kind == BC_DIRICHLET ? G.feq[side][part][i] : s[r];
        }
    }
}

// NP pairs of rows.
template <int TM, int NP>
__global__ void __launch_bounds__(kStripThreads, 16 / kStripWarps)
    k_strip(const BatchProb* __restrict__ probs, const StripWarp* __restrict__ warps, int rounds, int nsteps,
            int ns_max, long long* level_ptr, unsigned* bar_count, unsigned* bar_gen, unsigned* ticket,
            unsigned* status) {
    __shared__ Model<F2> sM[kStripWarps];
    // edge columns on their way to the neighbouring warps, by step parity:
    // [0] lane 1's, [1] lane 30's
    __shared__ Column<NP> sE[2][kStripWarps][2];
    // the column beside the left and the right ghost column, or the ghost
    // column itself where it stays the same; then room for split sides'
    __shared__ Column<NP> sX[kStripWarps][2], sY[kStripWarps][2];
    __shared__ int sRound;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const long long level0 = *(volatile long long*)level_ptr;
    unsigned bits = 0;
    // More rounds than CTAs: each CTA draws its next round while it works on
    // one (an SM does not share its issue slots evenly between its CTAs).
    // Every CTA draws until it gets one past the last, rounds + gridDim.x
    // tickets a pass in all.
    const bool drawn = rounds > (int)gridDim.x;
    unsigned base = 0;
    int done = 0, loaded = -1;
    while (done < nsteps) {
        int n = min(ns_max, nsteps - done);
        if ((n & 1) == 0) --n;  // odd: level + n lies in the other level buffer
        const long long level = level0 + done;
        const bool last = done + n == nsteps;
        if (drawn) {
            if (threadIdx.x == 0) sRound = (int)(atomicAdd(ticket, 1u) - base);
            __syncthreads();
        }
        // (unsigned: a launch that follows one that gave up may find the barrier's
        // count in between, and a ticket drawn beside one that has been taken back
        // to zero, which must not be a round)
        for (int round = drawn ? sRound : (int)blockIdx.x; (unsigned)round < (unsigned)rounds;) {
            const StripWarp W = warps[(size_t)round * kStripWarps + w];
            const bool busy = W.prob >= 0;
            const BatchProb& P = probs[busy ? W.prob : 0];
            const Grid<float>& G = P.G;
            const int nx = G.nx, col = W.col0 + lane;
            const size_t pl = (size_t)G.plane, row = (size_t)G.row;
            // ghost columns of this warp: the left one in lane 0, the right one in lane gr
            const bool has_left = busy && W.col0 < 0;
            const int gr = nx - W.col0;
            const bool has_right = busy && gr < 32;
            const int rule_l = has_left ? side_rule(G, S_LEFT, 2 * NP) : 0;
            const int rule_r = has_right ? side_rule(G, S_RIGHT, 2 * NP) : 0;
            // columns to store: not the copies of the neighbouring warps' columns
            const bool mine = busy && col >= W.c0 && col < W.c1 && !(lane == 0 && (W.links & 1)) &&
                              !(lane == 31 && (W.links & 2));
            F2 f[9][NP];
            {
                const float* in = P.f[(int)(level & 1)] + row + (size_t)(col + PADX);
                const bool in_range = busy && col <= nx;
#pragma unroll
                for (int i = 0; i < 9; ++i)
#pragma unroll
                    for (int k = 0; k < NP; ++k) {
                        const float* p = in + i * pl + 2 * k * row;
                        f[i][k] = in_range ? pair(__ldcg(p), __ldcg(p + row)) : bcast(1.0f);
                    }
            }
            int next = rounds;
            if (drawn && threadIdx.x == 0) next = (int)(atomicAdd(ticket, 1u) - base);
            if (loaded != round) {  // the windows' constants, by their first warps, while the columns arrive
                if (busy && !(W.links & 1)) {
                    const float* m = reinterpret_cast<const float*>(&P.M);
                    F2* d = reinterpret_cast<F2*>(&sM[W.slot]);
                    for (int q = lane; q < kModelWords; q += 32) d[q] = bcast(__ldg(m + q));
                }
                __syncthreads();
                loaded = round;
            }
            const Model<F2>& M = sM[W.slot];
            if (has_left && lane == 0 && rule_l == BC_DIRICHLET) sX[w][0].put(f);
            if (has_right && lane == gr && rule_r == BC_DIRICHLET) sX[w][1].put(f);
            for (int j = 0; j < n; ++j) {
                if (busy) {
                    F2 acc[9][NP];
#pragma unroll
                    for (int k = 0; k < NP; ++k) {
                        F2 c[9], a[9], rho, ux, uy, T;
#pragma unroll
                        for (int i = 0; i < 9; ++i) c[i] = f[i][k];
                        moments<float, TM, F2>(c, M, rho, ux, uy, T);
                        if (mine)
                            bits |= health(lane0(rho), lane0(ux), lane0(uy), lane0(T)) |
                                    health(lane1(rho), lane1(ux), lane1(uy), lane1(T));
                        relaxation<float, TM, F2>(M, c, rho, ux, uy, T, a);
#pragma unroll
                        for (int i = 0; i < 9; ++i) acc[i][k] = a[i];
                    }
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        F2 o[NP];
#pragma unroll
                        for (int k = 0; k < NP; ++k) {
                            // rows 2k + 1, 2k + 2 and rows 2k - 1, 2k
                            const F2 up = pair(lane1(f[i][k]), lane0(f[i][(k + 1) % NP]));
                            const F2 dn = pair(lane1(f[i][(k + NP - 1) % NP]), lane0(f[i][k]));
                            o[k] = update(M, i, acc[i][k], f[i][k], shfl_down(f[i][k]), shfl_up(f[i][k]),
                                                     up, dn);
                        }
#pragma unroll
                        for (int k = 0; k < NP; ++k) f[i][k] = o[k];
                    }
                    if (has_left || has_right) {
                        if (has_left && lane == 1 && rule_l != BC_DIRICHLET) sX[w][0].put(f);
                        if (has_right && lane == gr - 1 && rule_r != BC_DIRICHLET) sX[w][1].put(f);
                        __syncwarp();
                        const bool left = has_left && lane == 0;
                        if (left || (has_right && lane == gr)) {
                            const Column<NP>& x = sX[w][left ? 0 : 1];
                            const int rule = left ? rule_l : rule_r;
                            if (rule < 0) {
                                Column<NP>& y = sY[w][left ? 0 : 1];
                                split_ghost<NP>(G, left ? S_LEFT : S_RIGHT, x, level + j + 1, y);
                                y.get(f);
                            } else {
                                x.get(f, rule == BC_REFLECT);
                            }
                        }
                        __syncwarp();
                    }
                }
                if (j + 1 < n) {
                    Column<NP>(&E)[kStripWarps][2] = sE[j & 1];
                    if (busy && (lane == 1 || lane == 30)) E[w][lane == 30].put(f);
                    __syncthreads();
                    if (busy && ((lane == 0 && (W.links & 1)) || (lane == 31 && (W.links & 2))))
                        (lane == 0 ? E[w - 1][1] : E[w + 1][0]).get(f);
                }
            }
            const bool ghost = (has_left && lane == 0 && W.c0 == 0) || (has_right && lane == gr && W.c1 == nx);
            if (mine || ghost) {
                float* out = P.f[(int)((level + n) & 1)] + (size_t)(col + PADX);
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    float* p = out + i * pl;
#pragma unroll
                    for (int k = 0; k < NP; ++k) {
                        p[(2 * k + 1) * row] = lane0(f[i][k]);
                        p[(2 * k + 2) * row] = lane1(f[i][k]);
                    }
                    // the ghost rows, which no pass reads, at the end of the launch
                    if (last && mine) {
                        p[0] = lane1(f[i][NP - 1]);
                        p[(2 * NP + 1) * row] = lane0(f[i][0]);
                    }
                }
            }
            if (!drawn) break;
            __syncthreads();  // the round's shared memory is no longer read
            if (threadIdx.x == 0) sRound = next;
            __syncthreads();
            round = sRound;
        }
        base += (unsigned)rounds + gridDim.x;
        if (!grid_barrier(bar_count, bar_gen, status)) return;
        done += n;
    }
    report(status, bits);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *level_ptr = level0 + nsteps;
        *ticket = 0u;
    }
}
}  // namespace

cudaError_t strip_set_wait_cycles(long long cycles) {
    return cudaMemcpyToSymbol(g_wait_cycles, &cycles, sizeof(cycles));
}

template <int TM>
cudaError_t launch_strip(const BatchProb* probs, const StripWarp* warps, int rounds, int rows, int nsteps, int ns,
                         long long* level, unsigned* bar_count, unsigned* bar_gen, unsigned* ticket, unsigned* status,
                         int grid, cudaStream_t st) {
    const void* kern = rows == 4 ? (const void*)k_strip<TM, 2> : (const void*)k_strip<TM, 1>;
    void* args[] = {(void*)&probs, (void*)&warps, (void*)&rounds, (void*)&nsteps, (void*)&ns,
                    (void*)&level, (void*)&bar_count, (void*)&bar_gen, (void*)&ticket, (void*)&status};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kStripThreads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelExC(&cfg, kern, args);
}

template <int TM>
int strip_max_grid(int rows) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (rows == 4)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_strip<TM, 2>, kStripThreads, 0);
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_strip<TM, 1>, kStripThreads, 0);
    return sms * per_sm;
}

#define LBM_STRIP_INST(TM)                                                                                       \
    template cudaError_t launch_strip<TM>(const BatchProb*, const StripWarp*, int, int, int, int, long long*,    \
                                          unsigned*, unsigned*, unsigned*, unsigned*, int, cudaStream_t);        \
    template int strip_max_grid<TM>(int);
LBM_STRIP_INST(T_INT32)
LBM_STRIP_INST(T_INT64)
LBM_STRIP_INST(T_DF)
LBM_STRIP_INST(T_CONS)
#undef LBM_STRIP_INST

}  // namespace lbm
