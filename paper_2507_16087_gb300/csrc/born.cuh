// born.cuh -- kernels of the split-preconditioned Born iteration.
//
// One iteration of eq. BornAlt / Algorithm 1 (Stanziola et al.),
//     z = (L+I)^-1 (B x + y),   x <- x + nu B (z - x),   B = I - V,
// on a D-dim grid (D = 2, 3) with C = D+1 components.
//
// (L+I)^-1 couples the components per wavenumber by App. B.1's matrix
//     [ (a1 + l1)/l1 I        i t / sqrt(l1 l2)  ]
//     [ i t^H / sqrt(l1 l2)   (a2 + l2)/l2       ] ,   t_eta = k_eta e^{i k_eta dx/2}.
// Eliminating the velocity leaves ONE scalar per wavenumber: with
// (u, p) = (L+I)^-1 (v, r) and c1 = i sqrt(l1 l2), c2 = l2 (a1 + l1), c3 = (a1 + l1)(a2 + l2),
//     b   = r + sum_eta tm_eta v_eta,       tm_eta = -(c1 / c2) conj(t_eta)
//     p   = c2 b / (|k|^2 + c3)
//     u_eta = Pu v_eta + td_eta p,          Pu = l1 / (a1 + l1),  td_eta = -Pu c1 / (l1 l2) t_eta .
// tm_eta and td_eta depend on k_eta only and Pu not on k, so
//   * the sum b is built up axis by axis: once a velocity component and the partial sum are transformed along
//     axis eta, tm_eta v_eta is added and that component needs no further transform;
//   * Pu v_eta is added in real space (v = B x + y is there anyway), and td_eta p splits off the pressure at
//     the inverse transform of axis eta.
// The fields carried between the kernels are q (partial sum, later the pressure) in component slot D of w and the
// velocity components not yet merged (later the split-off gradients) in their own slots; slot 0 is used by rows apart only
// (k_rows):
//     rows     update of iteration k, then B x + y and the forward x transform: p and u_x merge into q
//     axis2 +  forward y transform (3D): u_y merges into q               3 fields in, 2 out
//     last2    forward transform of the last axis, the scalar solve, inverse transform: 2 fields in, 2 out
//     axis2 -  inverse y transform (3D): the y gradient splits off       2 fields in, 3 out
// i.e. 18 one-dimensional transforms and 160 B/voxel of w traffic a 3D float32 iteration where carrying the C
// components through every transform takes 24 and 256 B/voxel (2D: 10 and 64 B/voxel instead of 12 and 96).
// The adjoint [(L+I)^-1]^H is the same scheme with the constants conjugated.
//
// The scaled operator A_s x = L x + V x of a residual needs no 3-D transform at all: L's off-diagonal blocks are
// i t_eta / sqrt(l1 l2) per axis, so each is a 1-D transform pair along its own axis (k_deriv2, k_rows_op).
//
// Field layout: [C][n2][n1][n0] interleaved complex, x fastest.
// Medium layout: rs[eta][N] = (S+ rho)_eta / lambda1, kp[N] = 1/(rho c0^2 lambda2),
// et[N] = 2 alpha c0 / omega; gamma from per-axis tables at centres (gc) and
// at the staggered points (gs).  V is never stored: per voxel
//   v_eta = rs_eta * gamma_eta - a1/lambda1 + i (rs_eta omega)    ... minus i Im(a1)/lambda1
//   v_p   = kp [(gamma + et omega) + i (omega - gamma et)] - a2/lambda2
// (eq. LV with q = (i omega + gamma)/(rho c^2), c^2 of eq. 118).
#pragma once
#include <type_traits>

#include "fft.cuh"

namespace cbs {

// row kernel: start of a block of iterations, update + start of the next iteration (with / without the norms of
// the update), last update of a block, plain forward transform (no B, no y), plain (L+I)^-1 output
enum RowsMode { ROWS_FWD = 0, ROWS_FUSED = 1, ROWS_FUSED_NORM = 2, ROWS_INV = 3, ROWS_COPY = 4, ROWS_GREEN = 5 };
enum OpMode { OP_RESID = 0, OP_APPLY = 1 };

struct Dims {
    int D;          // 2 or 3
    int n0, n1, n2; // extents (n2 = 1 in 2D)
    long long N;    // voxels
};

template <typename R> struct Medium {
    const R* rs[3];
    const R* kp;
    const R* et;
    const R* gc[3];
    const R* gs[3];
    R omega;
    R a1r, a1i, a2r, a2i;  // a_j / lambda_j
};

// constants of (L+I)^-1, forward or adjoint (see the top of this file)
template <typename R> struct Symbol {
    cplx<R> Pu;            // lambda1 / (a1 + lambda1)
    cplx<R> c3;            // (a1 + lambda1)(a2 + lambda2)
    cplx<R> cs;            // lambda2 (a1 + lambda1) / N  (inverse-transform normalisation included)
    const cplx<R>* tm[3];  // merge factors per axis
    const cplx<R>* td[3];  // split factors per axis
    const R* k2[3];        // k_eta^2
};

// off-diagonal factors of L per axis, i t_eta / (sqrt(lambda1 lambda2) n_eta) (the 1-D transforms' normalisation
// included), negated for the adjoint
template <typename R> struct LOp {
    const cplx<R>* it[3];
};

// Per-row view of B = 1 - v for component c (conj for the adjoint).  Along a
// row only x varies, so the gamma terms of the other axes are row constants.
template <typename R> struct RowB {
    const R* g0;  // gamma along x: staggered table for u_x, centre table otherwise
    R grest;      // gamma contributions of y (and z)
    const R* m0;  // rs_c (velocity) or kp (pressure), at the row start
    const R* m1;  // et (pressure), at the row start
    bool pres;
};

template <typename R>
__device__ __forceinline__ RowB<R> row_B(const Medium<R>& M, int D, int c, int i1, int i2, long long vbase)
{
    RowB<R> rb;
    rb.pres = (c == D);
    rb.g0 = (c == 0) ? M.gs[0] : M.gc[0];
    R g = (c == 1) ? __ldg(M.gs[1] + i1) : __ldg(M.gc[1] + i1);
    if (D == 3) g += (c == 2) ? __ldg(M.gs[2] + i2) : __ldg(M.gc[2] + i2);
    rb.grest = g;
    const R* rsc = (c == 0) ? M.rs[0] : ((c == 1) ? M.rs[1] : M.rs[2]);
    rb.m0 = (rb.pres ? M.kp : rsc) + vbase;
    rb.m1 = M.et + vbase;
    return rb;
}

template <typename R>
__device__ __forceinline__ cplx<R> born_B(const Medium<R>& M, const RowB<R>& rb, int i0, bool adj)
{
    const R g = __ldg(rb.g0 + i0) + rb.grest;
    R vr, vi;
    if (!rb.pres) {
        const R r = __ldg(rb.m0 + i0);
        vr = r * g - M.a1r;
        vi = r * M.omega - M.a1i;
    } else {
        const R k = __ldg(rb.m0 + i0), e = __ldg(rb.m1 + i0);
        vr = k * (g + e * M.omega) - M.a2r;
        vi = k * (M.omega - g * e) - M.a2i;
    }
    return mk<cplx<R>, R>((R)1 - vr, adj ? vi : -vi);
}

// Programmatic dependent launch: every kernel of an iteration waits in grid_wait for the kernel before it, and only
// after that lets the one after it be scheduled.  So when a kernel's blocks start, everything up to the kernel before
// the one before it is complete and visible; only what the direct predecessor writes has to wait.
// The trigger comes before a block's last stores: the next kernel's blocks then find free SMs and start evenly.  Given
// right after the wait it packs them onto the SMs that finish first (64^3 23.6 against 20.9 us an iteration, 512^2 19.3
// against 15.7, 512^3 8.7 against 7.5 ms); only where neither kernel fills the SMs does the earlier start gain (early_next in
// launch.cuh; float64 kernels are not launched this way, see kDependent there).
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_trigger() { asm volatile("griddepcontrol.launch_dependents;"); }
constexpr int kSMs = 152;
template <typename R> __device__ __forceinline__ void grid_trigger_if(int early)  // (predicated: a branch here splits the loads that follow)
{
    if constexpr (sizeof(R) == 4)
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "setp.ne.s32 p, %0, 0;\n\t"
            "@p griddepcontrol.launch_dependents;\n\t}" ::"r"(early));
}

template <int T> struct RowSync {
    __device__ __forceinline__ void operator()() const
    {
        if constexpr (T <= 32) __syncwarp();
        else __syncthreads();
    }
};
struct BlockSync {
    __device__ __forceinline__ void operator()() const { __syncthreads(); }
};

// Block-wide sum of two values; thread 0 writes them to out[0..1].  Warps sum
// in the accumulator type A (float32 for the float32 path: float64 arithmetic
// is scarce on this GPU), the per-warp sums are combined in float64.
template <typename A> __device__ __forceinline__ void block_sum2(A a_in, A b_in, double* out)
{
    __shared__ double red[2][32];
    A aa = a_in, bb = b_in;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        aa += __shfl_down_sync(0xffffffffu, aa, o);
        bb += __shfl_down_sync(0xffffffffu, bb, o);
    }
    double a = (double)aa, b = (double)bb;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) { red[0][w] = a; red[1][w] = b; }
    __syncthreads();
    if (w == 0) {
        const int nw = (blockDim.x + 31) >> 5;
        a = lane < nw ? red[0][lane] : 0.0;
        b = lane < nw ? red[1][lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_down_sync(0xffffffffu, a, o);
            b += __shfl_down_sync(0xffffffffu, b, o);
        }
        if (lane == 0) { out[0] = a; out[1] = b; }
    }
}


// a * b + c and a * real in the accumulate form
template <typename CT> __device__ __forceinline__ CT cfma(CT a, CT b, CT c)
{
    c.x = fma(a.x, b.x, c.x);
    c.y = fma(a.x, b.y, c.y);
    c.x = fma(-a.y, b.y, c.x);
    c.y = fma(a.y, b.x, c.y);
    return c;
}

// ------------------------------------------------- bulk (TMA) staged rows
// cp.async.bulk copies of a block's contiguous rows into shared memory,
// completed on an mbarrier.  Every wait is bounded: on timeout the kernel
// records an error code in *err and leaves without touching its outputs.
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t phase)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(phase)
        : "memory");
    return ok != 0;
}

constexpr int kBulkWaitLimit = 1 << 22;  // try_wait rounds before a copy is declared lost
constexpr int kErrBulkTimeout = 1;

// true when the phase completed; false after kBulkWaitLimit rounds
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t phase, int limit = kBulkWaitLimit)
{
    for (int i = 0; i < limit; ++i)
        if (mbar_try_wait(bar, phase)) return true;
    return false;
}

// orders this thread's shared-memory accesses before later bulk copies that read or overwrite the buffer
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }


// ----------------------------------------------------------------- rows
// One transform unit is one x row of one component, done by T = NX / RX threads; a block holds U units.  Blocks
// of the first kind (b < npair) take U/2 rows of the pair (p, u_x): units [0, U/2) are the pressure's, the rest
// u_x's; blocks of the second kind take U rows of one other velocity component.  The rows are staged by one bulk
// copy each on mbarriers (w first, then x and the medium, then y) at the pitch of the transform's exchange, so the
// exchange runs in the staged w row and the rows that share a shared-memory phase lie on different banks.
// y lands in w's rows once the inverse transform has been read out of them (ysep = 0: two field buffers a block,
// more blocks an SM) or in a buffer of its own, issued at the start (ysep = 1: small grids, where a block's
// chain of waits is the time); rows of 1024 and more float32 points have no such buffer (YREG).
// APART (2D): every block holds one unit, u_x's too.  Its row keeps its own slot 0; k_last2's MERGE_X merges and splits it,
// a factor a column there, so that no block waits for or reads another's row.  The two modes without B (ROWS_COPY, ROWS_GREEN) load straight from global memory.
template <typename R, int NX, int RX> struct RowCfg {
    static constexpr int T = NX / RX;
    static constexpr int SL = RowPad<cplx<R>, NX, T>::SL;        // row pitch of the field buffers (values)
    static constexpr int ML = (SL + 3) / 4 * 4;                  // row pitch of the medium buffers (reals)
    // 64 threads: many small blocks in different phases keep copies in flight (128 threads, both with 16 values: 63.8
    // against 62.1 us at 128^3, 421 against 410 us at 256^3)
    static constexpr int UMAX = 64 / T < 2 ? 2 : 64 / T;
    static constexpr int UMIN = 32 / T < 2 ? 2 : 32 / T;  // whole warps
    // float32 rows of 1024 and more points: an SM holds too few of their large blocks to hide a second copy's wait
    // behind each other, so y goes from global memory straight into registers (1024^2 36.7 -> 31.7, 2048^2 154 -> 129
    // us; shorter rows lose: 128^3 55.3 against 58.3, 256^3 400 against 428)
    static constexpr bool YREG = sizeof(R) == 4 && NX >= 1024;
    static constexpr int MAXT = UMAX * T;
    // float32: 128 registers a thread with 16 values, 88 with 12 (96^3 30.8 against 34.7 us at 128, 192^3 209 against 221),
    // 72 with 8 (80 from 256 points: 72 spills there)
    static constexpr int THREADS_SM = RX > 12 ? 512 : (RX > 8 ? 704 : (NX >= 256 ? 768 : 896));
    static constexpr int MINB = sizeof(R) == 4 ? THREADS_SM / MAXT : 1;
    // whether the mode's y may have a buffer of its own (ysep): the updates, unless y goes to registers
    __host__ __device__ static constexpr bool own_y(int mode)
    {
        return !YREG && (mode == ROWS_FUSED || mode == ROWS_FUSED_NORM || mode == ROWS_INV);
    }
    // shared memory of a block of U units: x, w (and y), the medium rows (three a pair row), three barriers; the two
    // modes without B take the exchange only
    __host__ __device__ static constexpr size_t smem(int U, int mode, bool ysep)
    {
        const size_t field = (size_t)U * SL * sizeof(cplx<R>);
        if (mode == ROWS_COPY || mode == ROWS_GREEN) return field;
        return field * (own_y(mode) && ysep ? 3 : 2) + (size_t)U / 2 * 3 * ML * sizeof(R) + 32;
    }
    // of a block of one unit of its own (APART): its field buffers, two medium rows, the barriers
    __host__ __device__ static constexpr size_t smem_apart(int mode)
    {
        const size_t field = SL * sizeof(cplx<R>);
        if (mode == ROWS_COPY || mode == ROWS_GREEN) return field;
        return field * (own_y(mode) ? 3 : 2) + (size_t)2 * ML * sizeof(R) + 32;
    }
};

// B = 1 - v from a voxel's medium values, m0 = rs_c (velocity, m1 = 0) or kp (pressure, m1 = et):
//   Re B = c.x - m0 (g + m1 omega),  Im B = c.y - m0 (omega - g m1)  with c = 1 + a / lambda; conj for the adjoint
template <typename R> struct UnitB {
    R cr, ci, om, so;  // c, omega, sign of the imaginary part times omega
    R si;              // +1, adjoint -1
};
template <typename R> __device__ __forceinline__ UnitB<R> unit_B(const Medium<R>& M, bool pres, bool adj)
{
    UnitB<R> u;
    u.si = adj ? (R)-1 : (R)1;
    u.cr = (R)1 + (pres ? M.a2r : M.a1r);
    u.ci = u.si * (pres ? M.a2i : M.a1i);
    u.om = M.omega;
    u.so = u.si * M.omega;
    return u;
}
template <bool PAIR, typename R> __device__ __forceinline__ cplx<R> voxel_B(const UnitB<R>& u, R g, R m0, R m1)
{
    if constexpr (PAIR) return mk<cplx<R>, R>(fma(-m0, fma(m1, u.om, g), u.cr), fma(-m0, fma(-g * u.si, m1, u.so), u.ci));
    else return mk<cplx<R>, R>(fma(-m0, g, u.cr), fma(-m0, u.so, u.ci));
}

// Bound by HBM where w does not fit in L2 (256^3: 402 us, 164 B/voxel at 6.8 TB/s; 512^3: 3.56 ms at 6.2 TB/s), by latency
// where it does (128^3: 55 us at 61 % of DRAM throughput, 26 warps an SM; stalls first on the staged copies).  The kernels it
// replaced, one per component: 60.9 us, 438 us, 3.94 ms.
template <typename R, int NX, int RX, int MODE, bool APART = false>
__global__ void __launch_bounds__(RowCfg<R, NX, RX>::MAXT, RowCfg<R, NX, RX>::MINB)
k_rows(Dims d, Medium<R> M, Symbol<R> Sy, cplx<R>* __restrict__ x, const cplx<R>* __restrict__ y,
       cplx<R>* __restrict__ w, const cplx<R>* __restrict__ tw, int npair, int nsingle, int ysep, int early, int adj, R nu,
       double* __restrict__ partials, int* err)
{
    using CT = cplx<R>;
    using Cfg = RowCfg<R, NX, RX>;
    constexpr int T = Cfg::T, SL = Cfg::SL, ML = Cfg::ML;
    constexpr int np = plan_npass(NX, RX);
    constexpr bool UPDATE = MODE == ROWS_FUSED || MODE == ROWS_FUSED_NORM || MODE == ROWS_INV;
    constexpr bool HAS_W = UPDATE || MODE == ROWS_GREEN;
    constexpr bool HAS_B = UPDATE || MODE == ROWS_FWD;  // B, y and the medium
    constexpr bool HAS_FWD = MODE == ROWS_FWD || MODE == ROWS_FUSED || MODE == ROWS_FUSED_NORM || MODE == ROWS_COPY;
    constexpr bool YREG = UPDATE && RowCfg<R, NX, RX>::YREG;
    constexpr bool NORM = MODE == ROWS_FUSED_NORM || MODE == ROWS_INV;
    extern __shared__ __align__(128) unsigned char smraw[];
    const int U = APART ? 1 : blockDim.x / T, H = U >> 1;
    const int E = U * SL;
    CT* xs = reinterpret_cast<CT*>(smraw);
    CT* ws = HAS_B ? xs + E : xs;
    const bool yown = Cfg::own_y(MODE) && ysep != 0;
    CT* ys = yown ? ws + E : ws;
    R* ms = reinterpret_cast<R*>(ws + (yown ? 2 * E : E));
    uint64_t* bar = reinterpret_cast<uint64_t*>(ms + (APART ? 2 : 3 * H) * ML);
    const int lu = APART ? 0 : threadIdx.x / T, t = APART ? threadIdx.x : threadIdx.x % T;
    const long long rpc = d.N / NX;  // rows per component
    const bool pair = !APART && (int)blockIdx.x < npair;
    const int per = pair ? H : U;
    int c, b = blockIdx.x;
    if (pair) {
        c = d.D;
    } else {
        b -= npair;
        c = (APART ? 0 : 1) + b / nsingle;
        b = b % nsingle;
    }
    const long long row0 = (long long)b * per;
    const int nrow = (int)(rpc - row0 < per ? rpc - row0 : per);
    const bool isx = pair && lu >= H;  // this unit is u_x's
    const int lrow = isx ? lu - H : lu;
    if (isx) c = 0;
    const bool valid = lrow < nrow;
    const bool pres = APART ? c == d.D : pair && !isx;
    const bool two_medium = pair || (APART && pres);  // et beside kp
    constexpr int nbar = UPDATE ? (YREG ? 2 : 3) : 1;
    const long long v0 = row0 * NX;  // first voxel of the block's rows
    const int cs = pair ? d.D : c;   // component (slot) of the block's first array
    constexpr uint32_t FB = NX * sizeof(CT), MB = NX * sizeof(R);
    // rows of one array into consecutive buffer rows, one copy a row, the copies spread over the block's threads
    auto rows_in = [&](auto* dst, const auto* src, int pitch, uint32_t bytes, uint64_t* on) {
        for (int k = threadIdx.x; k < nrow; k += blockDim.x) bulk_g2s(dst + k * pitch, src + (long long)k * NX, bytes, on);
    };
    // The wait for the kernel before, then the copies of w.  x was last written two kernels ago, y and the medium never
    // are, so on a small grid (ysep) their copies go first and are on the way during the wait; on a grid of many waves
    // w goes first, the transform waits for nothing else (512^3 3.54 against 3.64 ms, 2048^2 154 against 161 us).
    auto w_in = [&]() {
        grid_wait();
        grid_trigger_if<R>(early);
        if constexpr (UPDATE) rows_in(ws, w + (long long)cs * d.N + v0, SL, FB, bar);
    };
    auto y_in = [&](uint64_t* on) {
        rows_in(ys, y + (long long)cs * d.N + v0, SL, FB, on);
        if (pair) rows_in(ys + H * SL, y + v0, SL, FB, on);
    };
    if constexpr (HAS_B) {
        if (threadIdx.x == 0) {
            const uint32_t fb = (uint32_t)nrow * FB, mb = (uint32_t)nrow * MB, two = pair ? 2u : 1u;
            const uint32_t meds = pair ? 3u : (two_medium ? 2u : 1u);
            for (int k = 0; k < nbar; ++k) mbar_init(bar + k, 1);
            if constexpr (UPDATE) {
                mbar_expect_tx(bar, fb);
                mbar_expect_tx(bar + 1, two * fb + meds * mb);
                if constexpr (!YREG) mbar_expect_tx(bar + 2, two * fb);
            } else {
                mbar_expect_tx(bar, 2u * two * fb + meds * mb);
            }
        }
        __syncthreads();
        if (UPDATE && !yown) w_in();
        uint64_t* bx = UPDATE ? bar + 1 : bar;
        rows_in(xs, x + (long long)cs * d.N + v0, SL, FB, bx);
        if (pair) {
            rows_in(xs + H * SL, x + v0, SL, FB, bx);
            rows_in(ms, M.kp + v0, ML, MB, bx);
            rows_in(ms + H * ML, M.et + v0, ML, MB, bx);
            rows_in(ms + 2 * H * ML, M.rs[0] + v0, ML, MB, bx);
        } else if (APART && pres) {
            rows_in(ms, M.kp + v0, ML, MB, bx);
            rows_in(ms + ML, M.et + v0, ML, MB, bx);
        } else {
            rows_in(ms, (APART && c == 0 ? M.rs[0] : (c == 1 ? M.rs[1] : M.rs[2])) + v0, ML, MB, bx);
        }
        if (!UPDATE || yown) y_in(UPDATE ? bar + 2 : bar);
    }
    if (!UPDATE || yown) w_in();
    TwCache<NX, RX, CT> tc;
    tw_load<NX, RX, T>(tc, t, tw);
    const long long rest = row0 + (valid ? lrow : 0);
    const long long fbase = (long long)c * d.N + rest * NX;
    // a timed-out wait records the error, lets the block's copies land and leaves; the decision is block-uniform
    auto lost = [&](int k) -> bool {
        if (!__syncthreads_or(!mbar_wait_bounded(bar + k, 0))) return false;
        if (threadIdx.x == 0) {
            atomicExch(err, kErrBulkTimeout);
            for (int j = k; j < nbar; ++j) mbar_wait_bounded(bar + j, 0);
        }
        return true;
    };
    CT* row = ws + lu * SL;  // this unit's row: staged w (or y), and its exchange
    const CT* xr = xs + lu * SL + t;
    const CT* yr = ys + lu * SL + t;
    const R* m0r = ms + (isx ? 2 * H + lrow : lrow) * ML + t;
    const R* m1r = ms + ((APART ? 1 : H) + lrow) * ML + t;
    UnitB<R> ub{};
    const R* g0 = nullptr;
    R grest = (R)0;
    if constexpr (HAS_B) {
        const RowB<R> rb = row_B(M, d.D, c, (int)(rest % d.n1), (int)(rest / d.n1), 0);
        ub = unit_B(M, pres, adj != 0);
        g0 = rb.g0 + t;
        grest = rb.grest;
    }
    const R has_et = pres ? (R)1 : (R)0;
    auto B_at = [&](int o, auto is_pair) -> CT {  // o: compile-time offset from t
        const R g = __ldg(g0 + o) + grest;
        if constexpr (decltype(is_pair)::value) return voxel_B<true>(ub, g, m0r[o], has_et * m1r[o]);
        else return voxel_B<false>(ub, g, m0r[o], (R)0);
    };
    CT v[RX];
    if constexpr (HAS_W) {
        // u_x's units read the pressure's row too
        const CT* wr;
        if constexpr (UPDATE) {
            if (lost(0)) return;
            wr = ws + lrow * SL + t;
        } else {
            wr = w + (long long)cs * d.N + rest * NX + t;
        }
#pragma unroll
        for (int s = 0; s < RX; ++s) v[s] = wr[T * slot_q<NX, RX, 0>(s)];
        if (pair) {
            if (isx) {
#pragma unroll
                for (int s = 0; s < RX; ++s) v[s] = cmul(v[s], __ldg(Sy.td[0] + t + T * slot_q<NX, RX, 0>(s)));
            }
            __syncthreads();  // the rows are read before the exchange (or, unstaged, the output) reuses them
        }
        fft_run<NX, RX, +1, true>(v, row, 1, t, tw, tc, RowSync<T>());
        if constexpr (UPDATE) {
            // (the wait's barrier also ends every read of the exchange by the inverse transform)
            if (lost(1)) return;
            if (!YREG && !yown) {
                fence_proxy_async_smem();  // the generic-proxy accesses of the buffer come before the copies' writes
                y_in(bar + 2);
            }
            if (!YREG && lost(2)) return;
        }
    } else if constexpr (HAS_B) {
        if (lost(0)) return;
    }
    if constexpr (UPDATE) {
        R s0 = (R)0, s1 = (R)0;
        // the velocity's Pu (B x + y) in real space; the pressure has no such term
        const CT pu = pres ? mk<CT, R>((R)0, (R)0) : Sy.Pu;
        CT* xo = x + fbase + t;
        const CT* yg = YREG ? y + fbase + t : yr;
        auto update = [&](auto is_pair) {
#pragma unroll
            for (int s = 0; s < RX; ++s) {
                const int o = T * slot_q<NX, RX, np>(s);
                const CT bv = B_at(o, is_pair);
                const CT xv = xr[o], yv = yg[o];
                const CT wo = cfma(bv, xv, yv);                 // B x + y
                const CT zx = cfma(pu, wo, csub(v[s], xv));     // z - x
                const CT bn = cscale(bv, nu);
                const CT xn = cfma(bn, zx, xv);
                if (valid) xo[o] = xn;
                if constexpr (NORM) {
                    s0 += cabs2(cmul(bn, zx));  // (not xn - x: that has lost x's low bits)
                    s1 += cabs2(xn);
                }
                if constexpr (HAS_FWD) v[s] = cfma(bv, xn, yv);
            }
        };
        if (two_medium) update(std::true_type());
        else update(std::false_type());
        if constexpr (NORM) {
            if (!valid) { s0 = (R)0; s1 = (R)0; }
            block_sum2(s0, s1, partials + 2 * (long long)blockIdx.x);
        }
        if constexpr (HAS_FWD) permute_slots<NX, RX, np, 0>(v);  // same positions, entry order of the forward transform
    } else if constexpr (MODE == ROWS_FWD) {
#pragma unroll
        for (int s = 0; s < RX; ++s) {
            const int o = T * slot_q<NX, RX, 0>(s);
            v[s] = cfma(two_medium ? B_at(o, std::true_type()) : B_at(o, std::false_type()), xr[o], yr[o]);
        }
    } else if constexpr (MODE == ROWS_COPY) {
#pragma unroll
        for (int s = 0; s < RX; ++s) v[s] = x[fbase + t + T * slot_q<NX, RX, 0>(s)];
    } else {  // ROWS_GREEN (the 1 / N of the inverse transforms is in the symbol)
        const CT pu = pres ? mk<CT, R>((R)0, (R)0) : Sy.Pu;
        if (valid) {
#pragma unroll
            for (int s = 0; s < RX; ++s) {
                const long long f = fbase + t + T * slot_q<NX, RX, np>(s);
                w[f] = cfma(pu, x[f], v[s]);
            }
        }
    }
    if constexpr (HAS_FWD) {
        fft_run<NX, RX, -1, true>(v, row, 1, t, tw, tc, RowSync<T>());
        CT* wo = w + fbase + t;
        grid_trigger();
        if (pair) {  // q = p + tm_x u_x
            CT* h = ws + (isx ? lu : lu + H) * SL + t;
            __syncthreads();  // every exchange read is done
            if (isx) {
#pragma unroll
                for (int s = 0; s < RX; ++s) h[s * T] = cmul(v[s], __ldg(Sy.tm[0] + t + T * slot_q<NX, RX, np>(s)));
            }
            __syncthreads();
            if (isx || !valid) return;
#pragma unroll
            for (int s = 0; s < RX; ++s) wo[T * slot_q<NX, RX, np>(s)] = cadd(v[s], h[s * T]);
        } else if (valid) {
#pragma unroll
            for (int s = 0; s < RX; ++s) wo[T * slot_q<NX, RX, np>(s)] = v[s];
        }
    }
}

// ------------------------------------------------- strided axes, two transforms a thread
// A tile is COLS columns by all N points of the axis; a thread holds RA values of each of two transforms, so the
// two share every twiddle and the merge / split / scalar solve between them is register arithmetic.  Columns are
// flattened over the other axes, so small extents fill whole tiles.
template <typename R, int N, int RA, int COLS> struct PairCfg {
    static constexpr int T = N / RA;
    static constexpr int THREADS = T * COLS;
    static constexpr bool PADC = COLS * sizeof(cplx<R>) < 128;
    static constexpr int FSTRIDE = (PADC ? RowPad<cplx<R>, N, T>::pad(N - 1) + 1 : N) * COLS;  // values of one field's exchange
    static constexpr size_t SMEM = plan_npass(N, RA) > 1 ? 2 * (size_t)FSTRIDE * sizeof(cplx<R>) : 0;
    // float32: 128 registers a thread
    static constexpr int MINB = sizeof(R) == 4 ? (THREADS >= 512 ? 1 : 512 / THREADS) : 1;
    static_assert(THREADS % 32 == 0 && THREADS <= 1024, "pair tile shape");
};

// A thread's values of one column, position q of the thread at p + q st, into / out of the slot order of pass P.
// The addresses are formed again for the stores (opaque pointer): kept from the loads they would take two registers
// a value through the whole transform.
template <int N, int RA, int P, typename CT>
__device__ __forceinline__ void col_load(CT (&v)[RA], const CT* p, long long st)
{
#pragma unroll
    for (int q = 0; q < RA; ++q) {
        v[q_slot<N, RA, P>(q)] = *p;
        p += st;
    }
}
template <int N, int RA, int P, typename CT>
__device__ __forceinline__ void col_store(CT* p, long long st, const CT (&v)[RA])
{
    asm volatile("" : "+l"(p));
#pragma unroll
    for (int q = 0; q < RA; ++q) {
        *p = v[q_slot<N, RA, P>(q)];
        p += st;
    }
}

// y axis of a 3D field (16.9 and 16.4 us at 128^3, 108 and 112 us at 256^3, 5.0 and 6.1 TB/s; the four-component
// transforms it replaced 21.9 and 20.5, 198 and 199 us).  S = -1: blocks b < npair transform (q, u_y) and store q + tm_y u_y; S = +1: they read q
// only and store the inverse transforms of q and td_y q (slot 1).  The other blocks transform two u_z columns a
// thread (the column and the one half the columns further on).
template <typename R, int NA, int RA, int COLS, int S>
__global__ void __launch_bounds__(PairCfg<R, NA, RA, COLS>::THREADS, PairCfg<R, NA, RA, COLS>::MINB)
k_axis2(Dims d, cplx<R>* __restrict__ w, const cplx<R>* __restrict__ tw, const cplx<R>* __restrict__ tab, int npair, int early)
{
    using CT = cplx<R>;
    using Cfg = PairCfg<R, NA, RA, COLS>;
    constexpr int T = NA / RA;
    constexpr int np = plan_npass(NA, RA);
    extern __shared__ __align__(16) unsigned char smraw[];
    CT* sm = reinterpret_cast<CT*>(smraw);
    const int col = threadIdx.x % COLS, t = threadIdx.x / COLS;
    const int ncol = d.n0 * d.n2;
    const bool pair = (int)blockIdx.x < npair;
    int ca = (pair ? blockIdx.x : blockIdx.x - npair) * COLS + col;
    const bool valid = ca < (pair ? ncol : ncol / 2);
    if (!valid) ca = 0;
    const int cb = pair ? ca : ca + ncol / 2;
    const long long plane = (long long)d.n0 * d.n1;
    const long long oa = (long long)(ca / d.n0) * plane + ca % d.n0;
    const long long ob = (long long)(cb / d.n0) * plane + cb % d.n0;
    CT* a = w + (long long)(pair ? 3 : 2) * d.N + oa + (long long)t * d.n0;
    CT* b = w + (long long)(pair ? 1 : 2) * d.N + ob + (long long)t * d.n0;
    const long long st = (long long)T * d.n0;
    CT v[2][RA];
    grid_wait();
    grid_trigger_if<R>(early);
    col_load<NA, RA, 0>(v[0], a, st);
    if (S < 0 || !pair) {
        col_load<NA, RA, 0>(v[1], b, st);
    } else {
#pragma unroll
        for (int s = 0; s < RA; ++s) v[1][s] = cmul(v[0][s], __ldg(tab + t + T * slot_q<NA, RA, 0>(s)));
    }
    fft_run_multi<NA, RA, 2, S, Cfg::PADC>(v, sm + col, COLS, Cfg::FSTRIDE, t, tw, BlockSync());
    if (S < 0 && pair) {
#pragma unroll
        for (int s = 0; s < RA; ++s) v[0][s] = cfma(v[1][s], __ldg(tab + t + T * slot_q<NA, RA, np>(s)), v[0][s]);
    }
    grid_trigger();
    if (valid) {
        col_store<NA, RA, np>(a, st, v[0]);
        if (S > 0 || !pair) col_store<NA, RA, np>(b, st, v[1]);
    }
}

// Last axis: forward transforms of (q, u_last), b = q + tm u_last, p = cs b / (|k|^2 + c3), inverse transforms of p
// and td p.  grid: ceil(n0 n1 / COLS) (3D) or ceil(n0 / COLS) (2D).  MERGE_X (2D, rows apart): u_x comes in slot 0 and merges
// here, td_x p leaves there.
// Bound on chip, by exchanges, barriers and the first loads of a wave: 22 us at 128^3 (6 at L2 rate), 129 us at 256^3 and 1.45
// ms at 512^3 (79 and 632 us at HBM rate); holding all four components it took 40.5 us, 334 us and 3.24 ms.
template <typename R, int NL, int RL, int COLS, bool MERGE_X = false>
__global__ void __launch_bounds__(PairCfg<R, NL, RL, COLS>::THREADS, PairCfg<R, NL, RL, COLS>::MINB)
k_last2(Dims d, Symbol<R> Sy, cplx<R>* __restrict__ w, const cplx<R>* __restrict__ tw, int early)
{
    using CT = cplx<R>;
    using Cfg = PairCfg<R, NL, RL, COLS>;
    constexpr int T = NL / RL;
    constexpr int np = plan_npass(NL, RL);
    extern __shared__ __align__(16) unsigned char smraw[];
    CT* sm = reinterpret_cast<CT*>(smraw);
    const int col = threadIdx.x % COLS, t = threadIdx.x / COLS;
    const int ncol = d.D == 3 ? d.n0 * d.n1 : d.n0;
    int ci = blockIdx.x * COLS + col;
    const bool valid = ci < ncol;
    if (!valid) ci = 0;
    CT* a = w + (long long)d.D * d.N + ci + (long long)t * ncol;
    CT* b = w + (long long)(d.D - 1) * d.N + ci + (long long)t * ncol;
    const long long st = (long long)T * ncol;
    CT v[2][RL];
    grid_wait();
    if (sizeof(R) == 4 && early) grid_trigger();  // (a branch, not the predicated form: 137 against 151 us at 256^3)
    col_load<NL, RL, 0>(v[0], a, st);
    col_load<NL, RL, 0>(v[1], b, st);
    CT* ux = w + ci + (long long)t * ncol;
    if constexpr (MERGE_X) {
        CT u[RL];
        col_load<NL, RL, 0>(u, ux, st);
        const CT tx = __ldg(Sy.tm[0] + ci);
#pragma unroll
        for (int s = 0; s < RL; ++s) v[0][s] = cfma(u[s], tx, v[0][s]);
    }
    R k2c = Sy.c3.x;
    if (d.D == 3) k2c += __ldg(Sy.k2[0] + ci % d.n0) + __ldg(Sy.k2[1] + ci / d.n0);
    else k2c += __ldg(Sy.k2[0] + ci);
    const CT* tm = d.D == 3 ? Sy.tm[2] : Sy.tm[1];
    const CT* td = d.D == 3 ? Sy.td[2] : Sy.td[1];
    const R* k2l = d.D == 3 ? Sy.k2[2] : Sy.k2[1];
    fft_run_multi<NL, RL, 2, -1, Cfg::PADC>(v, sm + col, COLS, Cfg::FSTRIDE, t, tw, BlockSync());
#pragma unroll
    for (int s = 0; s < RL; ++s) {
        const int k = t + T * slot_q<NL, RL, np>(s);
        const CT bk = cfma(v[1][s], __ldg(tm + k), v[0][s]);
        const CT mu = mk<CT, R>(k2c + __ldg(k2l + k), Sy.c3.y);
        const R inv = (R)1 / cabs2(mu);
        const CT im = cmulc(mk<CT, R>(Sy.cs.x * inv, Sy.cs.y * inv), mu);
        const CT p = cmul(bk, im);
        v[0][s] = p;
        v[1][s] = cmul(p, __ldg(td + k));
    }
    // the thread owns the same positions after the forward transform; reorder its registers into the entry order
    permute_slots<NL, RL, np, 0>(v[0]);
    permute_slots<NL, RL, np, 0>(v[1]);
    fft_run_multi<NL, RL, 2, +1, Cfg::PADC>(v, sm + col, COLS, Cfg::FSTRIDE, t, tw, BlockSync());
    grid_trigger();
    if (valid) {
        col_store<NL, RL, np>(a, st, v[0]);
        col_store<NL, RL, np>(b, st, v[1]);
        if constexpr (MERGE_X) {
            const CT tx = __ldg(Sy.td[0] + ci);
#pragma unroll
            for (int s = 0; s < RL; ++s) v[1][s] = cmul(v[0][s], tx);
            col_store<NL, RL, np>(ux, st, v[1]);
        }
    }
}

// --------------------------------------------------------- the operator A_s x, axis by axis
// Off-diagonal part of L along one strided axis e (1 = y, 2 = z): g_e = F^-1(i g t F p) into slot e of w and
// d = F^-1(i g conj(t) F u_e) into slot D (added to it when `add`).  Columns as in k_axis2 / k_last2.
template <typename R, int N, int RA, int COLS>
__global__ void __launch_bounds__(PairCfg<R, N, RA, COLS>::THREADS, PairCfg<R, N, RA, COLS>::MINB)
k_deriv2(Dims d, LOp<R> L, const cplx<R>* __restrict__ x, cplx<R>* __restrict__ w, const cplx<R>* __restrict__ tw,
         int e, int add)
{
    using CT = cplx<R>;
    using Cfg = PairCfg<R, N, RA, COLS>;
    constexpr int T = N / RA;
    constexpr int np = plan_npass(N, RA);
    extern __shared__ __align__(16) unsigned char smraw[];
    CT* sm = reinterpret_cast<CT*>(smraw);
    const int col = threadIdx.x % COLS, t = threadIdx.x / COLS;
    const bool last = e == d.D - 1;
    const int ncol = last ? (d.D == 3 ? d.n0 * d.n1 : d.n0) : d.n0 * d.n2;
    const long long astride = last ? ncol : d.n0;
    int ci = blockIdx.x * COLS + col;
    const bool valid = ci < ncol;
    if (!valid) ci = 0;
    const long long o = (last ? (long long)ci : (long long)(ci / d.n0) * d.n0 * d.n1 + ci % d.n0) + t * astride;
    const long long oa = (long long)d.D * d.N + o, ob = (long long)e * d.N + o;
    const long long st = (long long)T * astride;
    CT v[2][RA];
    grid_wait();
    grid_trigger_if<R>(gridDim.x <= kSMs);
    col_load<N, RA, 0>(v[0], x + oa, st);
    col_load<N, RA, 0>(v[1], x + ob, st);
    fft_run_multi<N, RA, 2, -1, Cfg::PADC>(v, sm + col, COLS, Cfg::FSTRIDE, t, tw, BlockSync());
    const CT* it = e == 1 ? L.it[1] : L.it[2];
#pragma unroll
    for (int s = 0; s < RA; ++s) {
        const CT f = __ldg(it + t + T * slot_q<N, RA, np>(s));  // i g t
        v[0][s] = cmul(v[0][s], f);
        v[1][s] = cmul(v[1][s], mk<CT, R>(-f.x, f.y));  // i g conj(t) = -conj(i g t)
    }
    permute_slots<N, RA, np, 0>(v[0]);
    permute_slots<N, RA, np, 0>(v[1]);
    fft_run_multi<N, RA, 2, +1, Cfg::PADC>(v, sm + col, COLS, Cfg::FSTRIDE, t, tw, BlockSync());
    if (valid) {
        col_store<N, RA, np>(w + ob, st, v[0]);
        if (add) {
            col_load<N, RA, np>(v[0], w + oa, st);
#pragma unroll
            for (int s = 0; s < RA; ++s) v[1][s] = cadd(v[0][s], v[1][s]);
        }
        col_store<N, RA, np>(w + oa, st, v[1]);
    }
}

// x axis of the operator and its diagonal: blocks as in k_rows (pair blocks transform p and u_x, the others only
// combine; APART: 2D, one unit a block), w on entry the gradients / divergence of k_deriv2.
// OP_RESID: w <- y - A_s x, partial (|w|^2, |y|^2);  OP_APPLY: w <- A_s x, no partials.
template <typename R, int NX, int RX, bool APART = false>
__global__ void __launch_bounds__(RowCfg<R, NX, RX>::MAXT, RowCfg<R, NX, RX>::MAXT <= 128 ? 3 : 1)
k_rows_op(Dims d, Medium<R> M, LOp<R> L, const cplx<R>* __restrict__ x, const cplx<R>* __restrict__ y,
          cplx<R>* __restrict__ w, const cplx<R>* __restrict__ tw, int npair, int nsingle, int mode, int adj,
          double* __restrict__ partials)
{
    using CT = cplx<R>;
    using Cfg = RowCfg<R, NX, RX>;
    constexpr int T = Cfg::T, SL = Cfg::SL;
    constexpr int np = plan_npass(NX, RX);
    extern __shared__ __align__(128) unsigned char smraw[];
    CT* ex = reinterpret_cast<CT*>(smraw);  // U * SL
    const int U = APART ? 1 : blockDim.x / T, H = U >> 1;
    const int lu = APART ? 0 : threadIdx.x / T, t = APART ? threadIdx.x : threadIdx.x % T;
    const long long rpc = d.N / NX;
    const bool pair = !APART && (int)blockIdx.x < npair;
    const int per = pair ? H : U;
    int c, b = blockIdx.x;
    if (pair) {
        c = d.D;
    } else {
        b -= npair;
        c = (APART ? 0 : 1) + b / nsingle;
        b = b % nsingle;
    }
    const long long row0 = (long long)b * per;
    const int nrow = (int)(rpc - row0 < per ? rpc - row0 : per);
    bool isx = pair && lu >= H;
    const int lrow = isx ? lu - H : lu;
    if (isx) c = 0;
    const bool valid = lrow < nrow;
    const bool pres = APART ? c == d.D : pair && !isx;
    if (APART) isx = c == 0;
    const bool xd = pair || (APART && c != 1);  // an x derivative goes into this unit's row
    const long long rest = row0 + (valid ? lrow : 0);
    const int i1 = (int)(rest % d.n1), i2 = (int)(rest / d.n1);
    const long long vbase = rest * NX;
    const long long fbase = (long long)c * d.N + vbase;
    const long long fother = (pres ? 0 : (long long)d.D * d.N) + vbase;  // APART: the row whose x derivative comes here
    const RowB<R> rb = row_B(M, d.D, c, i1, i2, vbase);
    CT v[RX];
    grid_wait();
    grid_trigger_if<R>(gridDim.x <= kSMs);
    if (xd) {
        TwCache<NX, RX, CT> tc;
        tw_load<NX, RX, T>(tc, t, tw);
#pragma unroll
        for (int s = 0; s < RX; ++s) v[s] = x[(APART ? fother : fbase) + t + T * slot_q<NX, RX, 0>(s)];
        CT* row = ex + (size_t)lu * SL;
        fft_run<NX, RX, -1, true>(v, row, 1, t, tw, tc, RowSync<T>());
#pragma unroll
        for (int s = 0; s < RX; ++s) {
            CT f = __ldg(L.it[0] + t + T * slot_q<NX, RX, np>(s));  // i g t
            if (APART ? pres : isx) f.x = -f.x;
            v[s] = cmul(v[s], f);
        }
        permute_slots<NX, RX, np, 0>(v);
        fft_run<NX, RX, +1, true>(v, row, 1, t, tw, tc, RowSync<T>());
        // the pressure's gradient goes to u_x and u_x's divergence to the pressure (APART: transformed from the other's row)
        if constexpr (!APART) {
            __syncthreads();
#pragma unroll
            for (int s = 0; s < RX; ++s) row[s * T + t] = v[s];
            __syncthreads();
            const CT* o = ex + (size_t)(isx ? lu - H : lu + H) * SL + t;
#pragma unroll
            for (int s = 0; s < RX; ++s) v[s] = o[s * T];
        }
    }
    R s0 = (R)0, s1 = (R)0;
    if (valid) {
#pragma unroll
        for (int s = 0; s < RX; ++s) {
            const int i0 = t + T * slot_q<NX, RX, np>(s);
            const CT xv = x[fbase + i0];
            // the whole diagonal, a / lambda + v: rs (gamma + i omega), or kp ((gamma + et omega) + i (omega - gamma et))
            const R g = __ldg(rb.g0 + i0) + rb.grest, m0 = __ldg(rb.m0 + i0);
            CT dg;
            if (pres) {
                const R et = __ldg(rb.m1 + i0);
                dg = mk<CT, R>(m0 * fma(et, M.omega, g), m0 * fma(-g, et, M.omega));
            } else {
                dg = mk<CT, R>(m0 * g, m0 * M.omega);
            }
            if (adj) dg.y = -dg.y;
            CT a = mk<CT, R>((R)0, (R)0);
            if (!isx) a = w[fbase + i0];
            if (xd) a = cadd(a, v[s]);
            a = cfma(dg, xv, a);
            if (mode == OP_RESID) {
                const CT yv = y[fbase + i0];
                a = csub(yv, a);
                s0 += cabs2(a);
                s1 += cabs2(yv);
            }
            w[fbase + i0] = a;
        }
    }
    if (mode == OP_RESID) block_sum2(s0, s1, partials + 2 * (long long)blockIdx.x);
}

}  // namespace cbs
