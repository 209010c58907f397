// noalloc.cu -- (L+I)^-1 apply that allocates no device memory.
//
// Some callers cannot call cudaMalloc: code running inside another
// framework's memory pool or under a fixed memory budget, plug-ins that must
// not grow the process's device footprint, or processes where the CUDA
// allocator is locked down.  green_apply_noalloc serves them: the caller
// passes the input and output buffers, and every other piece of device memory
// the transform needs (twiddle and wavenumber tables) lives in the file-scope
// array below.  That array is part of the library image: every GPU that loads
// the library holds it (kNoAllocScratchDoubles * 8 bytes = 84 KiB) until the
// process exits.
//
// The kernels are the same ones green_apply runs for a solver on the
// staggered grid (App. B.1, the default grid kind); the output buffer doubles
// as the transform's work array.  The collocated grid kind is not offered
// here: its symbol uses i k in place of i k e^{i k dx / 2}.
#include <cuda_runtime.h>

#include <cmath>
#include <complex>
#include <mutex>
#include <string>

#include "cbs.h"
#include "launch.cuh"

namespace cbs {
CBS_EXTERN_LAUNCHERS(double)
void set_create_error(const std::string& msg);  // message returned by cbs_last_error(NULL)
}  // namespace cbs

using namespace cbs;

namespace {

constexpr int kMaxAxis = 512;                    // largest supported extent
constexpr long long kMaxVoxels = 1LL << 21;      // N <= 2,097,152 (e.g. 128^3, 512 x 64 x 64, 512 x 512)
constexpr int kTwOff = 0;                                   // double2 tw[3][kMaxAxis]
constexpr int kTmOff = kTwOff + 3 * kMaxAxis * 2;           // double2 tm[3][kMaxAxis]: merge factors
constexpr int kTdOff = kTmOff + 3 * kMaxAxis * 2;           // double2 td[3][kMaxAxis]: split factors
constexpr int kK2Off = kTdOff + 3 * kMaxAxis * 2;           // double  k2[3][kMaxAxis]
constexpr int kNoAllocScratchDoubles = kK2Off + 3 * kMaxAxis;

static __device__ __align__(256) double g_noalloc_scratch[kNoAllocScratchDoubles];

constexpr int kMaxDevices = 64;
std::mutex g_mu;
double* g_scratch_addr[kMaxDevices] = {};

// Device address of the scratch array on the current device.  The name
// g_noalloc_scratch in host code is only a host-side stand-in, so the address
// is looked up once per device with that device current (the first call on
// that device) and kept for the life of the process; a process that resets a
// device with cudaDeviceReset must not call this entry point on that device
// afterwards, since the kept address belonged to the destroyed context.
cudaError_t scratch_address(double** out)
{
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_mu);
    if (g_scratch_addr[dev] == nullptr) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return e;
        g_scratch_addr[dev] = static_cast<double*>(p);
    }
    *out = g_scratch_addr[dev];
    return cudaSuccess;
}

// per-axis twiddles exp(-2 pi i j / n), merge and split factors fm conj(t) and fd t of t = k e^{i k dx/2}, and k^2,
// with k = 2 pi fftfreq(n, dx), written into the scratch tables
__global__ void k_noalloc_tables(int n0, int n1, int n2, double dx, double2 fm, double2 fd, double* scratch)
{
    const int a = blockIdx.y;
    const int n = a == 0 ? n0 : (a == 1 ? n1 : n2);
    double2* tw = reinterpret_cast<double2*>(scratch + kTwOff) + a * kMaxAxis;
    double2* tm = reinterpret_cast<double2*>(scratch + kTmOff) + a * kMaxAxis;
    double2* td = reinterpret_cast<double2*>(scratch + kTdOff) + a * kMaxAxis;
    double* k2 = scratch + kK2Off + a * kMaxAxis;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        double s, c;
        sincospi(-2.0 * (double)j / (double)n, &s, &c);
        tw[j] = make_double2(c, s);
        const int f = (j < (n + 1) / 2) ? j : j - n;
        const double k = 2.0 * 3.14159265358979323846 * (double)f / ((double)n * dx);
        double sh, ch;
        sincos(0.5 * k * dx, &sh, &ch);
        tm[j] = cmul(fm, make_double2(k * ch, -k * sh));
        td[j] = cmul(fd, make_double2(k * ch, k * sh));
        k2[j] = k * k;
    }
}

cbs_status fail(cbs_status st, const std::string& msg)
{
    set_create_error("green_apply_noalloc: " + msg);
    return st;
}

}  // namespace

extern "C" {

cbs_status green_apply_noalloc(const cbs_grid* grid, double dx, const double* scalars, const void* in, void* out,
                               int adjoint, void* stream)
{
    if (!grid || !scalars || !in || !out) return fail(CBS_EINVAL, "NULL argument");
    if (in == out) return fail(CBS_EINVAL, "in and out must be different buffers");
    if (grid->ndim != 2 && grid->ndim != 3) return fail(CBS_EINVAL, "ndim must be 2 or 3");
    long long N = 1;
    int n[3] = {1, 1, 1};
    for (int a = 0; a < grid->ndim; ++a) {
        if (!size_supported(grid->n[a]) || grid->n[a] > kMaxAxis)
            return fail(CBS_EINVAL, "unsupported extent " + std::to_string((long long)grid->n[a]));
        n[a] = (int)grid->n[a];
        N *= grid->n[a];
    }
    if (N > kMaxVoxels)
        return fail(CBS_EINVAL, "grid of " + std::to_string(N) + " voxels exceeds the allocation-free maximum of " +
                                    std::to_string(kMaxVoxels));
    const double l1 = scalars[4], l2 = scalars[5];
    if (!(dx > 0) || !(l1 > 0) || !(l2 > 0) || !std::isfinite(l1) || !std::isfinite(l2))
        return fail(CBS_EINVAL, "dx, lambda1 and lambda2 must be positive");
    double* scratch = nullptr;
    cudaError_t e = scratch_address(&scratch);
    if (e != cudaSuccess) return fail(CBS_ECUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    cudaStream_t st = (cudaStream_t)stream;

    Plan<double> P{};
    P.d.D = grid->ndim;
    P.d.n0 = n[0];
    P.d.n1 = n[1];
    P.d.n2 = n[2];
    P.d.N = N;
    // (L+I)^-1 constants (App. B.1, a = a1, lambda_0 = lambda1, b = a2, lambda_1 = lambda2; top of born.cuh),
    // conjugated for the adjoint
    using cd = std::complex<double>;
    auto cj = [&](cd v) { return adjoint ? std::conj(v) : v; };
    auto d2 = [](cd v) { return make_double2(v.real(), v.imag()); };
    const cd a1l(scalars[0] + l1, scalars[1]), a2l(scalars[2] + l2, scalars[3]);
    const cd c1 = cj(cd(0.0, std::sqrt(l1 * l2))), c2 = cj(l2 * a1l), pu = cj(l1 / a1l);
    Symbol<double>& Y = P.Sy[adjoint ? 1 : 0];
    Y.Pu = d2(pu);
    Y.c3 = d2(cj(a1l * a2l));
    Y.cs = d2(c2 / (double)N);
    for (int a = 0; a < 3; ++a) {
        P.tw[a] = reinterpret_cast<const double2*>(scratch + kTwOff) + a * kMaxAxis;
        Y.tm[a] = reinterpret_cast<const double2*>(scratch + kTmOff) + a * kMaxAxis;
        Y.td[a] = reinterpret_cast<const double2*>(scratch + kTdOff) + a * kMaxAxis;
        Y.k2[a] = scratch + kK2Off + a * kMaxAxis;
    }
    k_noalloc_tables<<<dim3(4, 3), 128, 0, st>>>(n[0], n[1], n[2], dx, d2(-(c1 / c2)), d2(-pu * c1 / (l1 * l2)), scratch);
    e = cudaGetLastError();
    if (e == cudaSuccess)
        e = launch_green<double>(P, static_cast<const double2*>(in), static_cast<double2*>(out), adjoint ? 1 : 0, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return fail(CBS_ECUDA, std::string("CUDA error ") + cudaGetErrorString(e));
    return CBS_OK;
}

}  // extern "C"
