// lbm_aux.cu -- initialisation, ghost fill, moments output, FP64 conservation
// totals and interior pack/unpack kernels of liblbm.
#include "lbm_launch.h"

namespace lbm {

namespace {
constexpr int kThreads = 256;

inline unsigned blocks_for(long long n, int per) { return (unsigned)((n + per - 1) / per); }

// The kernels below give a thread V consecutive columns of a row, a run.
// Where the rows' runs nearly fill CTAs of 64 x 4, a CTA takes such a patch, so
// that no index is divided (a 64-bit division per element had cost more than
// the copy: see launch_pack).  Other grids -- narrow, or a row of little more
// than so many runs -- take the runs in the order of the rows, a thread's row
// and column from one division, in 32 bits where that is enough (4 x 100000,
// FP32: moments 23 us, initial levels 42, get_f 21; in patches 54, 141 and 67),
// in CTAs of one warp where there are few.
constexpr int kRunX = 64;
struct RunGrid {
    dim3 grid;
    int threads;
    bool patch;
};
inline RunGrid run_grid(long long columns, long long rows, int V) {
    const long long runs = (columns + V - 1) / V, padded = (runs + kRunX - 1) / kRunX * kRunX;
    constexpr int kRunY = kThreads / kRunX;
    const bool few = runs * rows <= 512LL * kThreads;
    if ((few ? 2 * padded <= 3 * runs : 5 * padded <= 6 * runs) && rows >= kRunY &&
        rows <= 65535LL * kRunY)
        return {dim3((unsigned)(padded / kRunX), blocks_for(rows, kRunY)), kThreads, true};
    const int threads = runs * rows <= 16384 ? 32 : kThreads;
    return {dim3(blocks_for(runs * rows, threads)), threads, false};
}
template <int V, bool kPatch>
__device__ __forceinline__ bool run_place(int columns, int rows, int& x, int& row) {
    const unsigned runs = ((unsigned)columns + V - 1) / V;
    if constexpr (kPatch) {
        const unsigned k = blockIdx.x * kRunX + threadIdx.x % kRunX;
        row = (int)(blockIdx.y * (kThreads / kRunX) + threadIdx.x / kRunX);
        x = (int)k * V;
        return k < runs && row < rows;
    } else {
        const unsigned long long total = (unsigned long long)runs * (unsigned)rows;
        const unsigned long long q = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
        if (q >= total) return false;
        if (total <= 0xffffffffull) {
            row = (int)((unsigned)q / runs);
            x = (int)((unsigned)q % runs) * V;
        } else {
            row = (int)(q / runs);
            x = (int)(q % runs) * V;
        }
        return true;
    }
}

inline bool aligned(const void* p, size_t bytes) { return reinterpret_cast<uintptr_t>(p) % bytes == 0; }

// V = 2 or 4 consecutive FP32 values as packed pairs.
template <int V>
struct Run {
    F2 h[V / 2];
    __device__ __forceinline__ float at(int j) const { return j & 1 ? lane1(h[j / 2]) : lane0(h[j / 2]); }
};
template <int V>
struct alignas(4 * V) RunVec {
    float v[V];
};
// From / to an array: one access (wide), or n <= V single ones (values past
// n repeat the first).
template <int V>
__device__ __forceinline__ Run<V> load_run(const float* p, bool wide, int n) {
    RunVec<V> r;
    if (wide) {
        r = *reinterpret_cast<const RunVec<V>*>(p);
    } else {
#pragma unroll
        for (int j = 0; j < V; ++j) r.v[j] = j < n ? p[j] : p[0];
    }
    Run<V> o;
#pragma unroll
    for (int k = 0; k < V / 2; ++k) o.h[k] = pair(r.v[2 * k], r.v[2 * k + 1]);
    return o;
}
template <int V>
__device__ __forceinline__ void store_run(float* p, const Run<V>& o, bool wide, int n) {
    RunVec<V> r;
#pragma unroll
    for (int j = 0; j < V; ++j) r.v[j] = o.at(j);
    if (wide) {
        *reinterpret_cast<RunVec<V>*>(p) = r;
    } else {
#pragma unroll
        for (int j = 0; j < V; ++j)
            if (j < n) p[j] = r.v[j];
    }
}
}  // namespace

// f = f^eq(rho, u, T) (Eqs. e16-e18) at each interior node, and the ghost
// cells of level 0 by the edge nodes (from the values just stored, read
// back).  FP32: V x-adjacent nodes per thread in packed arithmetic, V-wide
// accesses; wide: the fields allow them too.  HBM-bound on large grids (16 B
// in, 36 B out a node): the stores want 16 bytes, 44 us on the 4096 x 1024
// grid with V = 4 against 48 with one node a thread, its index divided, and
// the ghost cells in a launch of their own.  Latency-bound on small ones,
// where V = 2 has twice the threads: 256 tubes of 4 rows one after the other
// 1.7-1.9 ms against 2.1 (V = 4) and 2.4 (two launches each); a batch takes
// k_init_batch.
constexpr long long kInitWideNodes = 1 << 20;
// V x-adjacent nodes from (ix, iy) on, and the ghost cells they write.
template <int V>
__device__ __forceinline__ void init_run(float* __restrict__ f, const float* __restrict__ rho,
                                         const float* __restrict__ ux, const float* __restrict__ uy,
                                         const float* __restrict__ T, const Model<float>& M, const Grid<float>& G,
                                         bool wide, int ix, int iy) {
    const int n = min(V, G.nx - ix);
    const size_t pl = (size_t)G.plane;
    const size_t q = (size_t)iy * G.nx + ix;
    const Run<V> r = load_run<V>(rho + q, wide, n), u = load_run<V>(ux + q, wide, n),
                 w = load_run<V>(uy + q, wide, n), t = load_run<V>(T + q, wide, n);
    F2 fe[V / 2][9];
#pragma unroll
    for (int k = 0; k < V / 2; ++k) equilibrium_scaled<float, F2>(M, r.h[k], u.h[k], w.h[k], t.h[k], fe[k]);
    float* out = f + cell(G, ix, iy);  // 4 V-byte aligned: ix + PADX is a multiple of V
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        Run<V> o;
#pragma unroll
        for (int k = 0; k < V / 2; ++k) o.h[k] = fe[k][i];
        store_run<V>(out + i * pl, o, n == V, n);
    }
    if (ix == 0 || iy == 0 || ix + n == G.nx || iy == G.ny - 1) {
        for (int j = 0; j < n; ++j) {
            float v[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) v[i] = out[i * pl + j];
            write_ghosts(G, f, ix + j, iy, v, 0);
        }
    }
}

template <int V, bool kPatch>
__global__ void __launch_bounds__(kThreads) k_init32(float* __restrict__ f, const float* __restrict__ rho,
                                                     const float* __restrict__ ux, const float* __restrict__ uy,
                                                     const float* __restrict__ T, const Model<float> M,
                                                     const Grid<float> G, bool wide) {
    int ix, iy;
    if (run_place<V, kPatch>(G.nx, G.ny, ix, iy)) init_run<V>(f, rho, ux, uy, T, M, G, wide, ix, iy);
}

// A batch's problems, one 64 x 4 tile of its tile list a CTA, the arrays'
// addresses in the launch's parameters: 256 tubes 0.50 ms
// (the kinds of 1024 addresses looked up by the host), 1.9 with a launch and a
// clearing of the status word per problem.
__global__ void __launch_bounds__(128) k_init_batch(const __grid_constant__ BatchInit A,
                                                    const BatchProb* __restrict__ probs,
                                                    const int4* __restrict__ tiles, int t0, int p0) {
    const int4 t = tiles[t0 + blockIdx.x];
    const BatchProb& P = probs[t.x];
    const BatchInit::Fields& a = A.of[t.x - p0];
    if (t.y == 0 && t.z == 0 && threadIdx.x == 0 && threadIdx.y == 0) *a.status = 0u;
    const int ix = t.y + 2 * threadIdx.x, iy = t.z + threadIdx.y;
    if (ix >= P.G.nx || iy >= P.G.ny) return;
    const bool wide = P.G.nx % 2 == 0 && (((uintptr_t)a.in[0] | (uintptr_t)a.in[1] | (uintptr_t)a.in[2] |
                                           (uintptr_t)a.in[3]) & 7) == 0;
    init_run<2>(P.f[0], a.in[0], a.in[1], a.in[2], a.in[3], P.M, P.G, wide, ix, iy);
}

template <int V>
void init32(float* f, const float* rho, const float* ux, const float* uy, const float* T, const Model<float>& M,
            const Grid<float>& G, bool wide, cudaStream_t st) {
    const RunGrid R = run_grid(G.nx, G.ny, V);
    (R.patch ? k_init32<V, true> : k_init32<V, false>)<<<R.grid, R.threads, 0, st>>>(f, rho, ux, uy, T, M, G, wide);
}

// One node a thread: FP64, and FP32 on large grids whose fields do not allow
// 16-byte accesses (a run of four would be read value by value: 4095 x 1023 64
// us, 40 here).  FP64 takes the nodes in their order in one-warp CTAs, and on
// large grids leaves the ghost cells to a kernel of their own: 4096 x 1024 320
// us, in patches and with them 347.
template <typename S, bool kGhosts>
__global__ void __launch_bounds__(kThreads) k_init(S* __restrict__ f, const S* __restrict__ rho,
                                                   const S* __restrict__ ux, const S* __restrict__ uy,
                                                   const S* __restrict__ T, const Model<S> M, const Grid<S> G) {
    int ix, iy;
    if (!run_place<1, false>(G.nx, G.ny, ix, iy)) return;
    const size_t q = (size_t)iy * G.nx + ix;
    S fe[9];
    equilibrium(M, rho[q], ux[q], uy[q], T[q], fe);
    const size_t c = cell(G, ix, iy);
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i * (size_t)G.plane + c] = fe[i];
    if constexpr (!kGhosts) return;
    if (ix == 0 || iy == 0 || ix == G.nx - 1 || iy == G.ny - 1) write_ghosts(G, f, ix, iy, fe, 0);
}

template <typename S>
cudaError_t launch_init(S* f, const S* rho, const S* ux, const S* uy, const S* T,
                        const Model<S>& M, const Grid<S>& G, cudaStream_t st) {
    if constexpr (sizeof(S) == 4) {
        auto wide = [&](int V) {
            return G.nx % V == 0 && aligned(rho, 4 * V) && aligned(ux, 4 * V) && aligned(uy, 4 * V) && aligned(T, 4 * V);
        };
        const bool large = (long long)G.nx * G.ny >= kInitWideNodes;
        if (!large)
            init32<2>(f, rho, ux, uy, T, M, G, wide(2), st);
        else if (wide(4))
            init32<4>(f, rho, ux, uy, T, M, G, true, st);
        else
            k_init<S, true><<<blocks_for((long long)G.nx * G.ny, kThreads), kThreads, 0, st>>>(f, rho, ux, uy, T, M, G);
    } else if ((long long)G.nx * G.ny >= kInitWideNodes) {
        k_init<S, false><<<blocks_for((long long)G.nx * G.ny, 32), 32, 0, st>>>(f, rho, ux, uy, T, M, G);
        return launch_fill_ghosts<S>(f, G, 0, st);
    } else {
        k_init<S, true><<<blocks_for((long long)G.nx * G.ny, 32), 32, 0, st>>>(f, rho, ux, uy, T, M, G);
    }
    return cudaGetLastError();
}

cudaError_t launch_init_batch(const BatchInit& args, const BatchProb* probs, const int4* tiles, int t0, int ntiles,
                              int p0, cudaStream_t st) {
    k_init_batch<<<ntiles, dim3(32, 4), 0, st>>>(args, probs, tiles, t0, p0);
    return cudaGetLastError();
}

// Every edge node writes the ghost cells it is responsible for (the same rule
// the step kernel applies to its output level).
template <typename S>
__global__ void k_fill_ghosts(S* __restrict__ f, const Grid<S> G, long long level) {
    const long long total = 2LL * G.nx + 2LL * G.ny;
    const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (q >= total) return;
    int ix, iy;
    if (q < G.nx) {
        ix = (int)q, iy = 0;
    } else if (q < 2LL * G.nx) {
        ix = (int)(q - G.nx), iy = G.ny - 1;
    } else if (q < 2LL * G.nx + G.ny) {
        ix = 0, iy = (int)(q - 2LL * G.nx);
    } else {
        ix = G.nx - 1, iy = (int)(q - 2LL * G.nx - G.ny);
    }
    const size_t c = cell(G, ix, iy);
    S v[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) v[i] = f[i * (size_t)G.plane + c];
    write_ghosts(G, f, ix, iy, v, level);
}

template <typename S>
cudaError_t launch_fill_ghosts(S* f, const Grid<S>& G, long long level, cudaStream_t st) {
    const long long total = 2LL * G.nx + 2LL * G.ny;
    k_fill_ghosts<S><<<blocks_for(total, kThreads), kThreads, 0, st>>>(f, G, level);
    return cudaGetLastError();
}

// Moments of a level.  FP32: two x-adjacent nodes per thread in packed
// arithmetic, 8-byte accesses; wide: the outputs allow them.  Near the HBM
// bound (36 B in, 16 B out a node) in the modes with few operations, also
// issue-bound with the double-float sum.  4096 x 1024: 43.3 us (double-float)
// and 35.7 (total energy), as with one node a thread; 1024 x 256 with the
// FP64 sum 10.0, one node a thread and its index divided 16.9.  Four nodes a
// thread: 59.9 and 47.5 (too few warps for their registers).
// (CTAs an SM: the FP64 sum spills in the 48 registers of five)
template <int TM, bool kPatch>
__global__ void __launch_bounds__(kThreads, TM == T_INT64 ? 4 : TM != T_CONS ? 5 : kPatch ? 8 : 6) k_moments32(const float* __restrict__ f, float* __restrict__ rho,
                                                        float* __restrict__ ux, float* __restrict__ uy,
                                                        float* __restrict__ T, const Model<float> M,
                                                        const Grid<float> G, unsigned* status, bool wide) {
    int ix, iy;
    unsigned bits = 0;
    if (run_place<2, kPatch>(G.nx, G.ny, ix, iy)) {
        const int n = min(2, G.nx - ix);
        const size_t pl = (size_t)G.plane;
        const float* in = f + cell(G, ix, iy);  // 8-byte aligned
        F2 v[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = load_run<2>(in + i * pl, n == 2, n).h[0];
        Run<2> r, u, w, t;
        moments<float, TM, F2>(v, M, r.h[0], u.h[0], w.h[0], t.h[0]);
        // the second lane of a last odd node repeats the first
        bits |= health(r.at(0), u.at(0), w.at(0), t.at(0)) | health(r.at(1), u.at(1), w.at(1), t.at(1));
        const size_t q = (size_t)iy * G.nx + ix;
        if (rho) store_run<2>(rho + q, r, wide, n);
        if (ux) store_run<2>(ux + q, u, wide, n);
        if (uy) store_run<2>(uy + q, w, wide, n);
        if (T) store_run<2>(T + q, t, wide, n);
    }
    report(status, bits);
}

__global__ void __launch_bounds__(32) k_moments64(const double* __restrict__ f, double* __restrict__ rho,
                                                        double* __restrict__ ux, double* __restrict__ uy,
                                                        double* __restrict__ T, const Model<double> M,
                                                        const Grid<double> G, unsigned* status) {
    int ix, iy;
    unsigned bits = 0;
    if (run_place<1, false>(G.nx, G.ny, ix, iy)) {
        const size_t c = cell(G, ix, iy);
        double v[9], r, u, w, t;
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = f[i * (size_t)G.plane + c];
        moments<double, T_PLAIN>(v, M, r, u, w, t);
        bits |= health(r, u, w, t);
        const size_t q = (size_t)iy * G.nx + ix;
        if (rho) rho[q] = r;
        if (ux) ux[q] = u;
        if (uy) uy[q] = w;
        if (T) T[q] = t;
    }
    report(status, bits);
}

template <typename S, int TM>
cudaError_t launch_moments(const S* f, S* rho, S* ux, S* uy, S* T, const Model<S>& M,
                           const Grid<S>& G, unsigned* status, cudaStream_t st) {
    if constexpr (sizeof(S) == 4) {
        const bool wide = G.nx % 2 == 0 && aligned(rho, 8) && aligned(ux, 8) && aligned(uy, 8) && aligned(T, 8);
        const RunGrid R = run_grid(G.nx, G.ny, 2);
        (R.patch ? k_moments32<TM, true> : k_moments32<TM, false>)<<<R.grid, R.threads, 0, st>>>(
            f, rho, ux, uy, T, M, G, status, wide);
    } else {
        k_moments64<<<blocks_for((long long)G.nx * G.ny, 32), 32, 0, st>>>(f, rho, ux, uy, T, M, G, status);
    }
    return cudaGetLastError();
}

// ------------------------------------------------------ conservation totals
// FP64 totals of rho, rho ux, rho uy and E = sum f (v^2 + eta^2) over the
// interior.  Each CTA reduces a fixed, strided subset of the grid's units (a
// unit is a run of kConsSeg columns of one row) in a fixed order; the last
// CTA to finish adds the CTAs' partials in a fixed order, so the result does
// not depend on scheduling, and writes it with the health word straight to
// the caller's page-locked memory.  (With a second kernel and two
// copies back a call took 30 us on the smallest grids.)  On those the
// kernel's time is that of its FP64 instructions one after the other, 64 cycles
// each: the reductions share the totals out over the lanes, and an FP64 CTA
// has one warp to each quarter of its SM (400 x 4, us a call: FP64 15.3 against
// 21.0, FP32 15.9 against 18.5).
constexpr int kConsSeg = 512, kConsSeg64 = 128;
constexpr int kConsBlocks = 608;  // 4 per SM

// Grids of at most kConsNarrow columns: a unit is kConsSeg (FP64: kConsSeg64)
// places, 2^cons_shift columns of several rows (a row alone would leave most
// of a warp's lanes idle: 4 x 100000, us a call, FP32 44 against 274, FP64 46
// against 216).
constexpr int kConsNarrow = 64;
__host__ __device__ inline int cons_shift(int nx) {
    int s = 2;  // a run of four
    while ((1 << s) < nx) ++s;
    return s;
}

template <typename S>
int conservation_partials(const Grid<S>& G) {
    const int seg = sizeof(S) == 4 ? kConsSeg : kConsSeg64;
    long long units = (long long)G.ny * ((G.nx + seg - 1) / seg);
    if (G.nx <= kConsNarrow) {
        const int rows = seg >> cons_shift(G.nx);
        units = ((long long)G.ny + rows - 1) / rows;
    }
    return (int)(units < kConsBlocks ? units : kConsBlocks);
}

namespace {
// The nine sums of a set of populations, as totals.
__device__ __forceinline__ void totals_of(const Model<double>& M, const double (&v)[9], double (&t)[4]) {
    const double s14 = (v[1] + v[3]) + (v[2] + v[4]);
    const double s58 = (v[5] + v[7]) + (v[6] + v[8]);
    t[0] = v[0] + s14 + s58;
    t[1] = M.c1 * (v[3] - v[1]) + M.d * ((v[6] + v[7]) - (v[5] + v[8]));
    t[2] = M.c1 * (v[4] - v[2]) + M.d * ((v[7] + v[8]) - (v[5] + v[6]));
    t[3] = M.eta2 * v[0] + M.c1s * s14 + M.c2s * s58;
}

// Sum over the eight lanes that share a total.
__device__ __forceinline__ double sum8(double v) {
#pragma unroll
    for (int d = 4; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
    return v;
}
// Sums of four quantities over a warp: the lanes 8 q .. 8 q + 7 get the q-th.
// Halves of the warp first take two of the four each, quarters one: six
// additions, where four shuffle trees take twenty.
__device__ __forceinline__ double warp_totals(const double (&t)[4]) {
    const int lane = threadIdx.x & 31;
    const bool up = lane & 16, odd = lane & 8;
    const double a = (up ? t[2] : t[0]) + __shfl_xor_sync(0xffffffffu, up ? t[0] : t[2], 16);
    const double b = (up ? t[3] : t[1]) + __shfl_xor_sync(0xffffffffu, up ? t[1] : t[3], 16);
    return sum8((odd ? b : a) + __shfl_xor_sync(0xffffffffu, odd ? a : b, 8));
}

// Called by one whole warp of a CTA, with the CTA's q-th total in the lanes 8 q
// .. 8 q + 7: writes the partials, and in the last CTA the totals and the
// health word.  left: CTAs that have finished, zero between launches.
__device__ __forceinline__ void finish_totals(double t, double* __restrict__ partials, unsigned* left,
                                              const unsigned* status, double* out, unsigned* out_status) {
    const int lane = threadIdx.x & 31, q = lane >> 3, k = lane & 7;
    const int nb = gridDim.x;
    if (k == 0) {
        __stcg(partials + q * nb + blockIdx.x, t);
        __threadfence();
    }
    __syncwarp();
    unsigned last = 0;
    if (lane == 0) last = atomicAdd(left, 1u) == (unsigned)nb - 1;
    if (!__shfl_sync(0xffffffffu, last, 0)) return;
    __threadfence();
    double acc = 0.0;
    for (int b = k; b < nb; b += 8) acc += __ldcg(partials + q * nb + b);
    acc = sum8(acc);
    if (k == 0) out[q] = acc;
    if (lane == 0) {
        *out_status = *status;
        *left = 0;
    }
}

// Running sum of FP32 values as h + l + c: h and l take each value by TwoSum
// (exact), c collects what l rounds away, so the sum carries about 72 bits:
// more than an FP64 accumulator, on the FP32 pipe.
template <typename V>
struct Sum3 {
    V h{}, l{}, c{};
    __device__ __forceinline__ void add(V x) {
        V s, e, t, d;
        two_sum(h, x, s, e);
        two_sum(l, e, t, d);
        h = s;
        l = t;
        c = add_(c, d);
    }
    __device__ __forceinline__ void add(const Sum3& o) {
        V s, e, t, d, u, g;
        two_sum(h, o.h, s, e);
        two_sum(l, o.l, t, d);
        two_sum(t, e, u, g);
        h = s;
        l = u;
        c = add_(add_(c, o.c), add_(d, g));
    }
};
}  // namespace

// FP32 levels: 9 warps, warp i sums population i of the CTA's units with
// 16-byte loads and packed Sum3 accumulators, and only the CTA's nine sums
// become FP64.  HBM-bound: a call on 4096 x 1024 takes 48 us, 39 of them the kernel;
// FP64 adds of every value (33 FP64 instructions a node, at 1/64 of the FP32
// rate) took 330.  Sums
// that leave the FP32 range, and levels with infinities or NaN, are taken
// again in FP64 by the warp that saw one.
constexpr int kConsThreads32 = 9 * 32;
__global__ void __launch_bounds__(kConsThreads32, 4)
    k_cons32(const float* __restrict__ f, const Model<double> M, const Grid<float> G, double* __restrict__ partials,
             unsigned* left, const unsigned* status, double* out, unsigned* out_status) {
    __shared__ double sums[3][9];
    const int pop = threadIdx.x / 32, lane = threadIdx.x & 31;
    const int segs = (G.nx + kConsSeg - 1) / kConsSeg;
    const long long units = (long long)G.ny * segs;
    auto run_of = [&](long long u, int& n) {
        const int row = (int)(u / segs), x0 = (int)(u % segs) * kConsSeg;
        n = min(kConsSeg, G.nx - x0);
        return f + (size_t)(row + 1) * (size_t)G.row + (size_t)pop * (size_t)G.plane + (PADX + x0);  // 16-byte aligned
    };
    Sum3<F2> a, b;
    const bool narrow = G.nx <= kConsNarrow;
    const int shift = cons_shift(G.nx), unit_rows = kConsSeg >> shift;
    auto row_of = [&](long long r) {
        return f + (size_t)(r + 1) * (size_t)G.row + (size_t)pop * (size_t)G.plane + PADX;
    };
    for (long long r0 = (long long)blockIdx.x * unit_rows; r0 < G.ny && narrow; r0 += (long long)gridDim.x * unit_rows) {
        float4 v[kConsSeg / 128];
#pragma unroll
        for (int k = 0; k < kConsSeg / 128; ++k) {
            const int q = k * 128 + lane * 4, x = q & ((1 << shift) - 1);
            const long long r = r0 + (q >> shift);
            v[k] = float4{0.0f, 0.0f, 0.0f, 0.0f};
            if (r < G.ny && x < G.nx) {
                v[k] = __ldg(reinterpret_cast<const float4*>(row_of(r) + x));  // within the row's padding
                if (x + 1 >= G.nx) v[k].y = 0.0f;
                if (x + 2 >= G.nx) v[k].z = 0.0f;
                if (x + 3 >= G.nx) v[k].w = 0.0f;
            }
        }
#pragma unroll
        for (int k = 0; k < kConsSeg / 128; ++k) {
            a.add(pair(v[k].x, v[k].y));
            b.add(pair(v[k].z, v[k].w));
        }
    }
    for (long long u = blockIdx.x; u < units && !narrow; u += gridDim.x) {
        int n;
        const float* p = run_of(u, n);
        float4 v[kConsSeg / 128];
#pragma unroll
        for (int k = 0; k < kConsSeg / 128; ++k) {
            const int x = k * 128 + lane * 4;
            v[k] = x + 3 < n ? __ldg(reinterpret_cast<const float4*>(p + x)) : float4{0.0f, 0.0f, 0.0f, 0.0f};
        }
        float tail = 0.0f;
        if (lane < (n & 3)) tail = __ldg(p + (n & ~3) + lane);
#pragma unroll
        for (int k = 0; k < kConsSeg / 128; ++k) {
            a.add(pair(v[k].x, v[k].y));
            b.add(pair(v[k].z, v[k].w));
        }
        if (n & 3) a.add(pair(tail, 0.0f));
    }
    a.add(b);
    Sum3<float> s, r;
    s.h = lane0(a.h), s.l = lane0(a.l), s.c = lane0(a.c);
    r.h = lane1(a.h), r.l = lane1(a.l), r.c = lane1(a.c);
    s.add(r);
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        r.h = __shfl_down_sync(0xffffffffu, s.h, d);
        r.l = __shfl_down_sync(0xffffffffu, s.l, d);
        r.c = __shfl_down_sync(0xffffffffu, s.c, d);
        s.add(r);
    }
    // lane 0 holds the sum; anything not finite on the way has made it NaN or
    // infinite, or its error terms NaN
    const bool fine = isfinite(s.h) && isfinite(s.l) && isfinite(s.c);
    double part[3] = {(double)s.h, (double)s.l, (double)s.c};
    if (!__shfl_sync(0xffffffffu, (int)fine, 0)) {
        double acc = 0.0;
        for (long long r0 = (long long)blockIdx.x * unit_rows; r0 < G.ny && narrow;
             r0 += (long long)gridDim.x * unit_rows)
            for (long long r = r0; r < r0 + unit_rows && r < G.ny; ++r)
                for (int x = lane; x < G.nx; x += 32) acc += (double)row_of(r)[x];
        for (long long u = blockIdx.x; u < units && !narrow; u += gridDim.x) {
            int n;
            const float* p = run_of(u, n);
            for (int x = lane; x < n; x += 32) acc += (double)p[x];
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, d);
        part[0] = acc;
        part[1] = part[2] = 0.0;
    }
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < 3; ++k) sums[k][pop] = part[k];
    __syncthreads();
    if (pop == 0) {
        // linear in the sums: the totals of each part in a lane of its own
        double v[9], t[4];
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = lane < 3 ? sums[lane][i] : 0.0;
        totals_of(M, v, t);
        finish_totals(warp_totals(t), partials, left, status, out, out_status);
    }
}

// FP64 levels: one node per thread, FP64 sums of the pair differences and of
// the three speed classes (17 FP64 instructions a node; forming the totals
// node by node takes 27), combined once per thread.
constexpr int kConsThreads64 = 128;
__global__ void __launch_bounds__(kConsThreads64)
    k_cons64(const double* __restrict__ f, const Model<double> M, const Grid<double> G, double* __restrict__ partials,
             unsigned* left, const unsigned* status, double* out, unsigned* out_status) {
    __shared__ double sh[4][kConsThreads64 / 32];
    const int segs = (G.nx + kConsSeg64 - 1) / kConsSeg64;
    const long long units = (long long)G.ny * segs;
    const size_t pl = (size_t)G.plane;
    double s0 = 0.0, s14 = 0.0, s58 = 0.0, ax = 0.0, ay = 0.0, ar = 0.0, am = 0.0;
    auto node = [&](const double* p) {
        double v[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) v[i] = __ldg(p + i * pl);
        s0 += v[0];
        s14 += (v[1] + v[3]) + (v[2] + v[4]);
        s58 += (v[5] + v[7]) + (v[6] + v[8]);
        ax += v[3] - v[1];
        ay += v[4] - v[2];
        ar += v[7] - v[5];
        am += v[6] - v[8];
    };
    const bool narrow = G.nx <= kConsNarrow;
    if (narrow) {
        const int shift = cons_shift(G.nx), x = threadIdx.x & ((1 << shift) - 1), rows = kConsSeg64 >> shift;
        for (long long r = (long long)blockIdx.x * rows + (threadIdx.x >> shift); r < G.ny;
             r += (long long)gridDim.x * rows)
            if (x < G.nx) node(f + cell(G, x, (int)r));
    }
    for (long long u = blockIdx.x; u < units && !narrow; u += gridDim.x) {
        const int row = (int)(u / segs), x0 = (int)(u % segs) * kConsSeg64;
        const int n = min(kConsSeg64, G.nx - x0);
        const double* p = f + cell(G, x0, row);
        for (int x = threadIdx.x; x < n; x += kConsThreads64) node(p + x);
    }
    double t[4] = {s0 + s14 + s58, M.c1 * ax + M.d * (ar + am), M.c1 * ay + M.d * (ar - am),
                   M.eta2 * s0 + M.c1s * s14 + M.c2s * s58};
    const int warp = threadIdx.x / 32, lane = threadIdx.x & 31;
    const double sum = warp_totals(t);
    if ((lane & 7) == 0) sh[lane >> 3][warp] = sum;
    __syncthreads();
    if (warp == 0) {
        const double part = (lane & 7) < kConsThreads64 / 32 ? sh[lane >> 3][lane & 7] : 0.0;
        finish_totals(sum8(part), partials, left, status, out, out_status);
    }
}

template <typename S>
cudaError_t launch_conservation(const S* f, const Model<double>& M, const Grid<S>& G, double* partials,
                                unsigned* left, const unsigned* status, double* out, unsigned* out_status,
                                cudaStream_t st) {
    const int nb = conservation_partials(G);
    if constexpr (sizeof(S) == 4)
        k_cons32<<<nb, kConsThreads32, 0, st>>>(f, M, G, partials, left, status, out, out_status);
    else
        k_cons64<<<nb, kConsThreads64, 0, st>>>(f, M, G, partials, left, status, out, out_status);
    return cudaGetLastError();
}

// Sum of n doubles by one CTA: strided partial sums, then a fixed tree.
__global__ void __launch_bounds__(1024) k_sum(const double* __restrict__ v, int n, double* out,
                                              const unsigned* status, unsigned* out_status) {
    __shared__ double sh[32];
    double t = 0.0;
    for (int k = threadIdx.x; k < n; k += 1024) t += v[k];
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) t += __shfl_down_sync(0xffffffffu, t, s);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x / 32] = t;
    __syncthreads();
    if (threadIdx.x < 32) {
        t = sh[threadIdx.x];
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) t += __shfl_down_sync(0xffffffffu, t, s);
        if (threadIdx.x == 0) {
            *out = t;
            *out_status = *status;
        }
    }
}

cudaError_t launch_sum(const double* v, int n, double* out, const unsigned* status, unsigned* out_status,
                       cudaStream_t st) {
    k_sum<<<1, 1024, 0, st>>>(v, n, out, status, out_status);
    return cudaGetLastError();
}

// ----------------------------------------------------------- pack / unpack
// Interior of a level <-> dense 9 x ny x nx array (kUnpack: dense to level),
// one population row at a time in the level's order ([row][population]), V
// values per access: 16 bytes where the dense rows allow it, else one value.
template <typename S, int V, bool kUnpack, bool kPatch>
__global__ void __launch_bounds__(kThreads) k_pack(S* __restrict__ f, S* __restrict__ dense, const Grid<S> G) {
    struct alignas(V * sizeof(S)) Vec {
        S v[V];
    };
    int x, r;
    if (!run_place<V, kPatch>(G.nx, 9 * G.ny, x, r)) return;  // ny is at most 2^24
    const int iy = r / 9, i = r - iy * 9;
    const long long n = (long long)G.nx * G.ny;
    Vec* a = reinterpret_cast<Vec*>(f + (size_t)(iy + 1) * (size_t)G.row + (size_t)i * (size_t)G.plane + (PADX + x));
    Vec* b = reinterpret_cast<Vec*>(dense + i * n + (long long)iy * G.nx + x);
    if constexpr (kUnpack)
        *a = *b;
    else
        *b = *a;
}

// 4096 x 1024 in FP32 (302 MB moved): 50 us, against 218 with one element a
// thread and its row and population found by 64-bit divisions.
template <typename S, bool kUnpack>
cudaError_t launch_copy(S* f, S* dense, const Grid<S>& G, cudaStream_t st) {
    constexpr int V = 16 / sizeof(S);
    const bool wide = G.nx % V == 0 && aligned(dense, 16);
    const RunGrid R = run_grid(G.nx, 9LL * G.ny, wide ? V : 1);
    auto kern = wide ? (R.patch ? k_pack<S, V, kUnpack, true> : k_pack<S, V, kUnpack, false>)
                     : (R.patch ? k_pack<S, 1, kUnpack, true> : k_pack<S, 1, kUnpack, false>);
    kern<<<R.grid, R.threads, 0, st>>>(f, dense, G);
    return cudaGetLastError();
}

template <typename S>
cudaError_t launch_pack(const S* f, S* dense, const Grid<S>& G, cudaStream_t st) {
    return launch_copy<S, false>(const_cast<S*>(f), dense, G, st);
}

template <typename S>
cudaError_t launch_unpack(S* f, const S* dense, const Grid<S>& G, cudaStream_t st) {
    return launch_copy<S, true>(f, const_cast<S*>(dense), G, st);
}

#define LBM_INST(S)                                                                          \
    template cudaError_t launch_init<S>(S*, const S*, const S*, const S*, const S*,          \
                                        const Model<S>&, const Grid<S>&, cudaStream_t);      \
    template cudaError_t launch_fill_ghosts<S>(S*, const Grid<S>&, long long, cudaStream_t); \
    template int conservation_partials<S>(const Grid<S>&);                                   \
    template cudaError_t launch_conservation<S>(const S*, const Model<double>&,              \
                                                const Grid<S>&, double*, unsigned*,          \
                                                const unsigned*, double*, unsigned*,         \
                                                cudaStream_t);                               \
    template cudaError_t launch_pack<S>(const S*, S*, const Grid<S>&, cudaStream_t);         \
    template cudaError_t launch_unpack<S>(S*, const S*, const Grid<S>&, cudaStream_t);
LBM_INST(double)
LBM_INST(float)
#undef LBM_INST

#define LBM_MOM_INST(S, TM)                                                                                  \
    template cudaError_t launch_moments<S, TM>(const S*, S*, S*, S*, S*, const Model<S>&, const Grid<S>&, \
                                               unsigned*, cudaStream_t);
LBM_MOM_INST(double, T_PLAIN)
LBM_MOM_INST(float, T_INT32)
LBM_MOM_INST(float, T_INT64)
LBM_MOM_INST(float, T_DF)
LBM_MOM_INST(float, T_CONS)
#undef LBM_MOM_INST

}  // namespace lbm
