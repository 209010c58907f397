// launch.cuh -- host-side launchers of the Born kernels for one precision.
// Each launcher dispatches on the axis extent to the kernel instantiated for
// that size (the FFT plans are compile-time).  Included by exactly one
// translation unit per precision and kernel group (kernels_*.cu).
#pragma once
#include <cuda_runtime.h>

#include "born.cuh"

namespace cbs {

// Elements per thread of one transform.
// float32 rows: 8 values a thread up to 128 points (8*8*2 at 72 instead of 16*8 at 128 registers a thread: 55.4 instead of
// 59.5 us at 128^3), 16 above (256^3 401 against 421 us, 512^3 3.55 against 4.16 ms). 3*2^k rows: 12 (192^3 209 against 221 us with 24).
template <typename R> __host__ __device__ constexpr int r_rows(int n)
{
    return (n % 3 == 0) ? 12 : ((sizeof(R) == 4 && n >= 256) ? 16 : 8);
}
// strided axes (two transforms a thread): 16 values for float32 axes of 128 and more points, else 8; 3*2^k: 12 (8 values
// at 128^3 / 256^3 / 512^3: last axis 24.2 / 161 / 1581 us against 22.1 / 137 / 1471)
template <typename R> __host__ __device__ constexpr int r_axis(int n)
{
    return (n % 3 == 0) ? 12 : ((sizeof(R) == 4 && n >= 128) ? 16 : 8);
}
// (the last axis takes the other strided axis's split, whatever the number of components)
template <typename R> __host__ __device__ constexpr int r_last(int n, int = 2) { return r_axis<R>(n); }
// small grids: fewer values a thread, so that a transform has more threads.  float32 (see small_tiles): 8 at every 2^k
// extent.  float64 (see few_warps): 4, and 6 up to 48 points: an SM sub-partition issues one FP64 warp instruction in
// 64 cycles, so a grid of fewer warps than there are sub-partitions takes as long as one warp's instructions.
template <typename R> __host__ __device__ constexpr int r_tile(int n)
{
    return sizeof(R) == 4 ? ((n % 3 == 0) ? 12 : 8) : ((n % 3 == 0) ? (n <= 48 ? 6 : 12) : (n <= 512 ? 4 : 8));
}
// rows of small grids (see rows_tiny)
template <typename R> __host__ __device__ constexpr int r_rows_tile(int n)
{
    return sizeof(R) == 4 ? (n == 512 ? 8 : r_rows<R>(n)) : r_tile<R>(n);
}

__host__ __device__ constexpr int max_i(int a, int b) { return a > b ? a : b; }
// columns of a tile: whole 128-byte lines where a tile of two transforms leaves room for several blocks an SM (us of
// the last axis, columns: 128^3 24.2 / 22.1 / 25.4 with 8 / 16 / 32, 256^3 149 / 137 with 8 / 16, 512^3 2261 / 1471 /
// 1622 with 4 / 8 / 16, 1024^2 23.0 / 27.5 with 4 / 8, 2048^2 112 / 90 with 2 / 4)
template <typename R> __host__ __device__ constexpr int cols_big(int n)
{
    const int t = n / r_axis<R>(n);
    return sizeof(R) == 4 ? max_i(n <= 256 ? 16 : (n <= 512 ? 8 : 4), 128 / t)
                          // float64 is bound by the FP64 pipes: small blocks, spread evenly (64^3: last axis 52.7 us
                          // with 4 columns, 58.7 with 8; 1024^2 312 with 1, 359 with 2; 2048^2 1407 and 1335)
                          : max_i(n == 1024 ? 1 : 2, 32 / t);
}
// small grids: 32-byte rows (float64 16), as many blocks as that gives
template <typename R> __host__ __device__ constexpr int cols_small(int n)
{
    const int t = n / r_tile<R>(n);
    return max_i(sizeof(R) == 4 ? 4 : 1, 32 / t);
}

#define CBS_FOR_EACH_SIZE(X) X(8) X(12) X(16) X(24) X(32) X(48) X(64) X(96) X(128) X(192) X(256) X(512) X(1024) X(2048)

inline bool size_supported(long long n)
{
    switch (n) {
#define CBS_CASE(n) case n:
        CBS_FOR_EACH_SIZE(CBS_CASE)
#undef CBS_CASE
        return true;
    default:
        return false;
    }
}

template <typename R> struct Plan {
    Dims d;
    Medium<R> M;
    Symbol<R> Sy[2];       // (L+I)^-1: forward, adjoint
    LOp<R> L[2];           // L: forward, adjoint
    const cplx<R>* tw[3];  // twiddle table of each axis length
    int* err = nullptr;    // device error word of the staged copies' bounded waits
};

// One launch; `dependent`: the kernel may be scheduled while the one before it in the stream still runs (it waits in
// grid_wait).  Only for kernels whose predecessor is one of the kernels here.
template <typename Kern, typename... Args>
cudaError_t launch(Kern kern, long long grid, int threads, size_t smem, cudaStream_t st, bool dependent, Args... args)
{
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = dependent ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// float32 only: float64 blocks, bound by their SM's FP64 pipe, gain 1-4 % on small grids but 25 % is lost where the next
// kernel's blocks are packed onto the SMs that finish first (256^2: 73.5 against 58.7 us an iteration)
template <typename R> constexpr bool kDependent = sizeof(R) == 4;

constexpr int kWaveBlocks = 2 * kSMs;  // two blocks on every SM
constexpr int kApartN = 2048;          // row length of rows_apart
constexpr int kApartRows = 48;         // and the largest extent of its other axis (three blocks a row, an SM each)

// float64 grids whose threads, each with r values, make fewer warps than there are SM sub-partitions (4 an SM)
template <typename R> inline bool few_warps(long long values, int r)
{
    return sizeof(R) == 8 && values / r < 32LL * 4 * kSMs;
}

// transform units (x rows of one component) of a row block: as many as 64 threads hold, halved while the grid
// would leave SMs without two blocks
template <typename R, int N, int RX> inline int rows_units_n(const Dims& d)
{
    using Cfg = RowCfg<R, N, RX>;
    const long long units = (long long)(d.D + 1) * (d.N / N);
    int u = Cfg::UMAX;
    while (u > Cfg::UMIN && units / u < kWaveBlocks) u /= 2;
    return u;
}
// whether the row kernels take r_rows_tile values a thread on this grid: float64 where r_rows leaves too few warps,
// float32 512-point rows where all of them are on the SMs at once (512^2: 14.5 against 16.1 us an iteration)
template <typename R> inline bool rows_tiny(int n, const Dims& d)
{
    if (r_rows_tile<R>(n) >= r_rows<R>(n)) return false;
    const long long values = (long long)(d.D + 1) * d.N;
    return sizeof(R) == 8 ? few_warps<R>(values, r_rows<R>(n)) : values / r_rows<R>(n) <= 512LL * kSMs;
}
template <typename R, int N> inline bool rows_tiny(const Dims& d) { return rows_tiny<R>(N, d); }

struct RowGrid {
    int units, npair, nsingle, blocks;
};
template <typename R, int N> inline RowGrid row_grid(const Dims& d)
{
    RowGrid g;
    g.units = rows_tiny<R, N>(d) ? rows_units_n<R, N, r_rows_tile<R>(N)>(d) : rows_units_n<R, N, r_rows<R>(N)>(d);
    const long long rpc = d.N / N;
    g.npair = (int)((rpc + g.units / 2 - 1) / (g.units / 2));
    g.nsingle = (int)((rpc + g.units - 1) / g.units);
    g.blocks = g.npair + (d.D - 1) * g.nsingle;
    return g;
}

// Whether the small tile of an axis is another one at all, and for float32 of fewer columns: from 1024 points it has the
// big tile's columns, so it makes no more blocks, and its 1024-thread blocks spill (us an iteration: 2048 points 8 columns
// 23.2 against 19.1 with the big tile, 128 columns 29.2 against 25.1, 512 columns 53.2 against 47.5; 1024 points 64 columns
// 14.3 against 14.0, 512 columns 29.0 against 28.5).
template <typename R> constexpr bool has_small_tile(int n)
{
    return sizeof(R) == 4 ? cols_small<R>(n) < cols_big<R>(n)
                          : cols_small<R>(n) != cols_big<R>(n) || r_tile<R>(n) != r_axis<R>(n);
}
// whether a strided axis of N points and `columns` columns (of two transforms) takes the small tiles: float32 when the
// big ones leave SMs without a block (64^3, 256 tiles: 20.3 us an iteration with the big ones against 20.9; 512^2, 64
// tiles: 17.8 against 15.9), float64 when the big ones make too few warps
template <typename R> inline bool small_tiles(int n, long long columns)
{
    if (!has_small_tile<R>(n)) return false;
    if (sizeof(R) == 8) return few_warps<R>(columns * n, r_axis<R>(n));
    return (columns + cols_big<R>(n) - 1) / cols_big<R>(n) < kSMs;
}

// Whether a float32 kernel of `blocks` blocks lets the next one start right after its own wait (see grid_wait): with at most
// a block an SM itself, and where the next kernel's blocks, packed onto the SMs with room, don't crowd them: one warp an SM of
// a strided axis or six of the row kernel.  us an iteration, early / late.  Rows before a strided axis: 24 x 2048 (128 warps)
// 12.0 / 15.2, 48 x 1024 (128) 10.8 / 12.8, 96 x 1024 (256) 13.3 / 12.4, 96 x 2048 (512) 18.8 / 15.6.  Last axis before rows:
// 128^2 (192 warps) 7.4 / 8.4, 256^2 (384) 9.0 / 10.1, 96 x 512 (576) 10.1 / 10.9, 512 x 128 (768) 9.8 / 10.3, 192 x 512
// (1152) 13.3 / 11.3, 256 x 512 (1536) 12.1 / 10.0.
template <typename R> inline int early_next(const Dims& d, long long blocks, bool rows_next, int n, long long columns)
{
    if (sizeof(R) != 4 || blocks > kSMs) return 0;
    if (rows_next) {
        const int r = rows_tiny<R>(d.n0, d) ? r_rows_tile<R>(d.n0) : r_rows<R>(d.n0);
        return (d.D + 1) * d.N / r <= 6 * 32 * kSMs;
    }
    const int r = small_tiles<R>(n, columns) ? r_tile<R>(n) : r_axis<R>(n);
    return columns * (n / r) <= 32 * kSMs;
}
// columns (of two transforms) of the y axis of a 3D field and of the last axis
inline long long axis_columns(const Dims& d) { return (long long)d.n0 * d.n2 * 3 / 2; }
inline long long last_columns(const Dims& d) { return d.D == 3 ? (long long)d.n0 * d.n1 : d.n0; }
template <typename R> inline int early_axis(const Dims& d, long long blocks) { return early_next<R>(d, blocks, false, d.n1, axis_columns(d)); }
template <typename R> inline int early_last(const Dims& d, long long blocks)
{
    return early_next<R>(d, blocks, false, d.D == 3 ? d.n2 : d.n1, last_columns(d));
}
template <typename R> inline int early_rows(const Dims& d, long long blocks) { return early_next<R>(d, blocks, true, 0, 0); }

// 2D grids of few long rows: a block, and so an SM, for every row of a component in place of one for a row of the pressure and
// of u_x together, whose FP64 instructions (float64) or chain of waits (float32) is the time.  us an iteration, pairs / apart
// (with every component transformed by itself, as before the scalar form, in brackets): float64 8 x 2048 126 / 68 [79], 48 x
// 2048 143 / 86 [107]; float32 8 x 2048 10.4 / 7.8 [11.2], 48 x 2048 13.5 / 11.5 [12.9].  With more rows an SM has two
// of them either way, and the last axis of the pairs carries no third field (64 x 2048 144 [175]).
template <typename R> inline bool rows_apart(const Dims& d) { return d.D == 2 && d.n0 == kApartN && (d.D + 1) * d.n1 <= kSMs; }

// blocks of the row kernels (= norm partials of one iteration)
template <typename R> inline int rows_blocks(const Plan<R>& P)
{
    if (rows_apart<R>(P.d)) return (P.d.D + 1) * P.d.n1;
    switch (P.d.n0) {
#define CBS_CASE(n) case n: return row_grid<R, n>(P.d).blocks;
        CBS_FOR_EACH_SIZE(CBS_CASE)
#undef CBS_CASE
    default: return 0;
    }
}

constexpr size_t kMaxDynSmem = 226 * 1024;  // 227 KiB less the reduction scratch

template <typename R, int N, int RX, int MODE>
cudaError_t rows_nm(const Plan<R>& P, cplx<R>* x, const cplx<R>* y, cplx<R>* w, int adj, R nu, double* partials,
                    cudaStream_t st)
{
    using Cfg = RowCfg<R, N, RX>;
    auto kern = k_rows<R, N, RX, MODE>;
    constexpr bool kOwnY = Cfg::own_y(MODE) && Cfg::smem(Cfg::UMAX, MODE, true) < kMaxDynSmem;
    // once per process, thread-safe (function-local static)
    static const cudaError_t attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                         (int)Cfg::smem(Cfg::UMAX, MODE, kOwnY));
    if (attr != cudaSuccess) return attr;
    const RowGrid g = row_grid<R, N>(P.d);
    // a grid of few blocks an SM gives y a buffer of its own, its copy in flight from the start (us an iteration: 128^2
    // 7.4 against 8.1, 256^2 8.9 against 9.5, 512^2 with 768 blocks 14.0 against 14.5); above that the room costs more
    // blocks than the wait does time (192^3 rows 331 against 296 us).  No block takes a buffer that its mode or row
    // length does not use: with y's, 1024- and 2048-point rows ran three and one blocks an SM in place of four and two
    // (96 x 2048 22.1 against 18.6 us an iteration, 512 x 2048 60.9 against 50.6)
    const int ysep = kOwnY && g.blocks <= 4 * kWaveBlocks ? 1 : 0;
    // the modes that start a chain follow other work (x and y may have just been written)
    return launch(kern, g.blocks, g.units * Cfg::T, Cfg::smem(g.units, MODE, ysep != 0), st,
                  kDependent<R> && MODE != ROWS_FWD && MODE != ROWS_COPY, P.d, P.M, P.Sy[adj ? 1 : 0], x, y, w, P.tw[0], g.npair, g.nsingle, ysep,
                  P.d.D == 3 ? early_axis<R>(P.d, g.blocks) : early_last<R>(P.d, g.blocks), adj, nu, partials, P.err);
}

template <typename R, int N, int RX, int MODE>
cudaError_t rows_apart_nm(const Plan<R>& P, cplx<R>* x, const cplx<R>* y, cplx<R>* w, int adj, R nu, double* partials,
                          cudaStream_t st)
{
    using Cfg = RowCfg<R, N, RX>;
    auto kern = k_rows<R, N, RX, MODE, true>;
    static const cudaError_t attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::smem_apart(MODE));
    if (attr != cudaSuccess) return attr;
    const int blocks = (P.d.D + 1) * P.d.n1;
    return launch(kern, blocks, Cfg::T, Cfg::smem_apart(MODE), st, kDependent<R> && MODE != ROWS_FWD && MODE != ROWS_COPY, P.d, P.M,
                  P.Sy[adj ? 1 : 0], x, y, w, P.tw[0], 0, P.d.n1, 1, early_last<R>(P.d, blocks), adj, nu, partials, P.err);
}

template <typename R, int N, int RX, int MODE>
cudaError_t rows_any_nm(const Plan<R>& P, cplx<R>* x, const cplx<R>* y, cplx<R>* w, int adj, R nu, double* partials,
                        cudaStream_t st)
{
    if constexpr (N == kApartN) {
        if (rows_apart<R>(P.d)) return rows_apart_nm<R, N, RX, MODE>(P, x, y, w, adj, nu, partials, st);
    }
    return rows_nm<R, N, RX, MODE>(P, x, y, w, adj, nu, partials, st);
}

template <typename R, int N, int RX>
cudaError_t rows_rx(const Plan<R>& P, cplx<R>* x, const cplx<R>* y, cplx<R>* w, int mode, int adj, R nu,
                    double* partials, cudaStream_t st)
{
    switch (mode) {
    case ROWS_FWD: return rows_any_nm<R, N, RX, ROWS_FWD>(P, x, y, w, adj, nu, partials, st);
    case ROWS_FUSED: return rows_any_nm<R, N, RX, ROWS_FUSED>(P, x, y, w, adj, nu, partials, st);
    case ROWS_FUSED_NORM: return rows_any_nm<R, N, RX, ROWS_FUSED_NORM>(P, x, y, w, adj, nu, partials, st);
    case ROWS_INV: return rows_any_nm<R, N, RX, ROWS_INV>(P, x, y, w, adj, nu, partials, st);
    case ROWS_COPY: return rows_any_nm<R, N, RX, ROWS_COPY>(P, x, y, w, adj, nu, partials, st);
    case ROWS_GREEN: return rows_any_nm<R, N, RX, ROWS_GREEN>(P, x, y, w, adj, nu, partials, st);
    default: return cudaErrorInvalidValue;
    }
}

template <typename R, int N>
cudaError_t rows_n(const Plan<R>& P, cplx<R>* x, const cplx<R>* y, cplx<R>* w, int mode, int adj, R nu,
                   double* partials, cudaStream_t st)
{
    if constexpr (r_rows_tile<R>(N) < r_rows<R>(N)) {
        if (rows_tiny<R, N>(P.d)) return rows_rx<R, N, r_rows_tile<R>(N)>(P, x, y, w, mode, adj, nu, partials, st);
    }
    return rows_rx<R, N, r_rows<R>(N)>(P, x, y, w, mode, adj, nu, partials, st);
}

// row kernels (see RowsMode); ROWS_COPY and ROWS_GREEN only read x
template <typename R>
cudaError_t launch_rows(const Plan<R>& P, cplx<R>* x, const cplx<R>* y, cplx<R>* w, int mode, int adj, R nu,
                        double* partials, cudaStream_t st)
{
    switch (P.d.n0) {
#define CBS_CASE(n) case n: return rows_n<R, n>(P, x, y, w, mode, adj, nu, partials, st);
        CBS_FOR_EACH_SIZE(CBS_CASE)
#undef CBS_CASE
    default: return cudaErrorInvalidValue;
    }
}

template <typename R, int N, int RX>
cudaError_t rows_op_rx(const Plan<R>& P, const cplx<R>* x, const cplx<R>* y, cplx<R>* w, int mode, int adj,
                       double* partials, cudaStream_t st)
{
    using Cfg = RowCfg<R, N, RX>;
    if constexpr (N == kApartN) {
        if (rows_apart<R>(P.d)) {
            auto kern = k_rows_op<R, N, RX, true>;
            constexpr size_t smem = Cfg::SL * sizeof(cplx<R>);
            static const cudaError_t attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (attr != cudaSuccess) return attr;
            return launch(kern, (P.d.D + 1) * P.d.n1, Cfg::T, smem, st, kDependent<R>, P.d, P.M, P.L[adj ? 1 : 0], x, y, w, P.tw[0],
                          0, P.d.n1, mode, adj, partials);
        }
    }
    auto kern = k_rows_op<R, N, RX>;
    constexpr int kMax = (int)((size_t)Cfg::UMAX * Cfg::SL * sizeof(cplx<R>));
    static const cudaError_t attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMax);
    if (attr != cudaSuccess) return attr;
    const RowGrid g = row_grid<R, N>(P.d);
    return launch(kern, g.blocks, g.units * Cfg::T, (size_t)g.units * Cfg::SL * sizeof(cplx<R>), st, kDependent<R>, P.d, P.M,
                  P.L[adj ? 1 : 0], x, y, w, P.tw[0], g.npair, g.nsingle, mode, adj, partials);
}

template <typename R, int N>
cudaError_t rows_op_n(const Plan<R>& P, const cplx<R>* x, const cplx<R>* y, cplx<R>* w, int mode, int adj,
                      double* partials, cudaStream_t st)
{
    if constexpr (r_rows_tile<R>(N) < r_rows<R>(N)) {
        if (rows_tiny<R, N>(P.d)) return rows_op_rx<R, N, r_rows_tile<R>(N)>(P, x, y, w, mode, adj, partials, st);
    }
    return rows_op_rx<R, N, r_rows<R>(N)>(P, x, y, w, mode, adj, partials, st);
}

// x axis and diagonal of the operator (after launch_deriv of the other axes)
template <typename R>
cudaError_t launch_rows_op(const Plan<R>& P, const cplx<R>* x, const cplx<R>* y, cplx<R>* w, int mode, int adj,
                           double* partials, cudaStream_t st)
{
    switch (P.d.n0) {
#define CBS_CASE(n) case n: return rows_op_n<R, n>(P, x, y, w, mode, adj, partials, st);
        CBS_FOR_EACH_SIZE(CBS_CASE)
#undef CBS_CASE
    default: return cudaErrorInvalidValue;
    }
}

template <typename R, int N, int RA, int COLS, int S> cudaError_t axis2_tile(const Plan<R>& P, cplx<R>* w, int adj, cudaStream_t st)
{
    using Cfg = PairCfg<R, N, RA, COLS>;
    auto kern = k_axis2<R, N, RA, COLS, S>;
    static const cudaError_t attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::SMEM);
    if (attr != cudaSuccess) return attr;
    const int ncol = P.d.n0 * P.d.n2;
    const int npair = (ncol + COLS - 1) / COLS, blocks = npair + (ncol / 2 + COLS - 1) / COLS;
    const Symbol<R>& Sy = P.Sy[adj ? 1 : 0];
    return launch(kern, blocks, Cfg::THREADS, Cfg::SMEM, st, kDependent<R>, P.d, w, P.tw[1], S < 0 ? Sy.tm[1] : Sy.td[1], npair,
                  S < 0 ? early_last<R>(P.d, blocks) : early_rows<R>(P.d, blocks));
}
template <typename R, int N, int S> cudaError_t axis2_n(const Plan<R>& P, cplx<R>* w, int adj, cudaStream_t st)
{
    constexpr int CB = cols_big<R>(N), CS = cols_small<R>(N);
    if constexpr (has_small_tile<R>(N)) {
        if (small_tiles<R>(N, axis_columns(P.d)))
            return axis2_tile<R, N, r_tile<R>(N), CS, S>(P, w, adj, st);
    }
    return axis2_tile<R, N, r_axis<R>(N), CB, S>(P, w, adj, st);
}

// y axis of a 3D field: sign -1 transforms forward and merges u_y, +1 transforms back and splits the y gradient off
template <typename R> cudaError_t launch_axis(const Plan<R>& P, cplx<R>* w, int sign, int adj, cudaStream_t st)
{
    switch (P.d.n1) {
#define CBS_CASE(n) case n: return sign < 0 ? axis2_n<R, n, -1>(P, w, adj, st) : axis2_n<R, n, +1>(P, w, adj, st);
        CBS_FOR_EACH_SIZE(CBS_CASE)
#undef CBS_CASE
    default: return cudaErrorInvalidValue;
    }
}

template <typename R, int N, int RL, int COLS, bool MERGE_X = false>
cudaError_t last2_tile(const Plan<R>& P, cplx<R>* w, int adj, cudaStream_t st)
{
    using Cfg = PairCfg<R, N, RL, COLS>;
    auto kern = k_last2<R, N, RL, COLS, MERGE_X>;
    static const cudaError_t attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::SMEM);
    if (attr != cudaSuccess) return attr;
    const long long blocks = (last_columns(P.d) + COLS - 1) / COLS;
    return launch(kern, blocks, Cfg::THREADS, Cfg::SMEM, st, kDependent<R>, P.d, P.Sy[adj ? 1 : 0], w, P.tw[P.d.D - 1],
                  P.d.D == 3 ? early_axis<R>(P.d, blocks) : early_rows<R>(P.d, blocks));
}
template <typename R, int N> cudaError_t last2_n(const Plan<R>& P, cplx<R>* w, int adj, cudaStream_t st)
{
    constexpr int CB = cols_big<R>(N), CS = cols_small<R>(N);
    if constexpr (N <= kApartRows) {  // (2048 columns of at most 48 points: the small tile's)
        if (rows_apart<R>(P.d)) return last2_tile<R, N, r_tile<R>(N), CS, true>(P, w, adj, st);
    }
    if constexpr (has_small_tile<R>(N)) {
        if (small_tiles<R>(N, last_columns(P.d))) return last2_tile<R, N, r_tile<R>(N), CS>(P, w, adj, st);
    }
    return last2_tile<R, N, r_last<R>(N), CB>(P, w, adj, st);
}

// last axis: forward transform, scalar solve, inverse transform
template <typename R> cudaError_t launch_last(const Plan<R>& P, cplx<R>* w, int adj, cudaStream_t st)
{
    switch (P.d.D == 3 ? P.d.n2 : P.d.n1) {
#define CBS_CASE(n) case n: return last2_n<R, n>(P, w, adj, st);
        CBS_FOR_EACH_SIZE(CBS_CASE)
#undef CBS_CASE
    default: return cudaErrorInvalidValue;
    }
}

template <typename R, int N, int RA, int COLS>
cudaError_t deriv_tile(const Plan<R>& P, const cplx<R>* x, cplx<R>* w, int e, int add, int adj, cudaStream_t st)
{
    using Cfg = PairCfg<R, N, RA, COLS>;
    auto kern = k_deriv2<R, N, RA, COLS>;
    static const cudaError_t attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::SMEM);
    if (attr != cudaSuccess) return attr;
    const int n[3] = {P.d.n0, P.d.n1, P.d.n2};
    const long long ncol = P.d.N / n[e];
    return launch(kern, (ncol + COLS - 1) / COLS, Cfg::THREADS, Cfg::SMEM, st, kDependent<R> && add != 0, P.d, P.L[adj ? 1 : 0], x, w, P.tw[e],
                  e, add);
}
template <typename R, int N>
cudaError_t deriv_n(const Plan<R>& P, const cplx<R>* x, cplx<R>* w, int e, int add, int adj, cudaStream_t st)
{
    constexpr int CB = cols_big<R>(N), CS = cols_small<R>(N);
    if constexpr (has_small_tile<R>(N)) {
        if (small_tiles<R>(N, P.d.N / N)) return deriv_tile<R, N, r_tile<R>(N), CS>(P, x, w, e, add, adj, st);
    }
    return deriv_tile<R, N, r_axis<R>(N), CB>(P, x, w, e, add, adj, st);
}

// off-diagonal part of L along the strided axis e (1 or 2), see k_deriv2
template <typename R>
cudaError_t launch_deriv(const Plan<R>& P, const cplx<R>* x, cplx<R>* w, int e, int add, int adj, cudaStream_t st)
{
    switch (e == 1 ? P.d.n1 : P.d.n2) {
#define CBS_CASE(n) case n: return deriv_n<R, n>(P, x, w, e, add, adj, st);
        CBS_FOR_EACH_SIZE(CBS_CASE)
#undef CBS_CASE
    default: return cudaErrorInvalidValue;
    }
}

// the whole (L+I)^-1 apply out = (L+I)^-1 x (out is also the work array; x != out)
template <typename R> cudaError_t launch_green(const Plan<R>& P, const cplx<R>* x, cplx<R>* out, int adj, cudaStream_t st)
{
    cplx<R>* xr = const_cast<cplx<R>*>(x);  // the two row modes only read it
    cudaError_t e = launch_rows<R>(P, xr, nullptr, out, ROWS_COPY, adj, (R)0, nullptr, st);
    if (e == cudaSuccess && P.d.D == 3) e = launch_axis<R>(P, out, -1, adj, st);
    if (e == cudaSuccess) e = launch_last<R>(P, out, adj, st);
    if (e == cudaSuccess && P.d.D == 3) e = launch_axis<R>(P, out, +1, adj, st);
    if (e == cudaSuccess) e = launch_rows<R>(P, xr, nullptr, out, ROWS_GREEN, adj, (R)0, nullptr, st);
    return e;
}

// out = y - A_s x (OP_RESID) or A_s x (OP_APPLY), norm partials of rows_blocks blocks (x != out)
template <typename R>
cudaError_t launch_operator(const Plan<R>& P, const cplx<R>* x, const cplx<R>* y, cplx<R>* out, int mode, int adj,
                            double* partials, cudaStream_t st)
{
    cudaError_t e = launch_deriv<R>(P, x, out, P.d.D - 1, 0, adj, st);
    if (e == cudaSuccess && P.d.D == 3) e = launch_deriv<R>(P, x, out, 1, 1, adj, st);
    if (e == cudaSuccess) e = launch_rows_op<R>(P, x, y, out, mode, adj, partials, st);
    return e;
}

// explicit instantiations: one translation unit per precision for the row kernels, one for the strided axes
#define CBS_ROW_LAUNCHERS(X, R)                                                                                      \
    X cudaError_t launch_rows<R>(const Plan<R>&, cplx<R>*, const cplx<R>*, cplx<R>*, int, int, R, double*, cudaStream_t); \
    X cudaError_t launch_rows_op<R>(const Plan<R>&, const cplx<R>*, const cplx<R>*, cplx<R>*, int, int, double*, cudaStream_t);
#define CBS_AXIS_LAUNCHERS(X, R)                                                                                     \
    X cudaError_t launch_axis<R>(const Plan<R>&, cplx<R>*, int, int, cudaStream_t);                                   \
    X cudaError_t launch_last<R>(const Plan<R>&, cplx<R>*, int, cudaStream_t);                                        \
    X cudaError_t launch_deriv<R>(const Plan<R>&, const cplx<R>*, cplx<R>*, int, int, int, cudaStream_t);
// declarations for translation units that only call the launchers
#define CBS_EXTERN_LAUNCHERS(R)                                                                                      \
    CBS_ROW_LAUNCHERS(extern template, R)                                                                            \
    CBS_AXIS_LAUNCHERS(extern template, R)

}  // namespace cbs
