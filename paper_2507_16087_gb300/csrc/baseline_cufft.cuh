// baseline_cufft.cuh -- the comparison build of the Born iteration: the same
// step (eq. BornAlt, the App. B.1 symbol) with the transforms done by cuFFT
// (batched complex-to-complex plans over the C components) and everything else
// by plain grid-stride pointwise kernels, one pass over the field each:
//     w = B x + y;  w = FFT(w);  w = G(k) w;  w = IFFT(w);  x += nu B (w - x)
// It exists to be timed beside the fused kernels; the solver never uses it.
#pragma once
#include "born.cuh"

namespace cbs {

__device__ __forceinline__ void voxel_coords(const Dims& d, long long v, int& i0, int& i1, int& i2)
{
    i0 = (int)(v % d.n0);
    const long long rest = v / d.n0;
    i1 = (int)(rest % d.n1);
    i2 = (int)(rest / d.n1);
}

// w = B x + y over all components
template <typename R>
__global__ void k_base_pre(Dims d, Medium<R> M, const cplx<R>* __restrict__ x, const cplx<R>* __restrict__ y,
                           cplx<R>* __restrict__ w, int adj)
{
    const long long n = (long long)(d.D + 1) * d.N;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i / d.N);
        const long long v = i % d.N;
        int i0, i1, i2;
        voxel_coords(d, v, i0, i1, i2);
        const RowB<R> rb = row_B(M, d.D, c, i1, i2, v - i0);
        w[i] = cadd(cmul(born_B(M, rb, i0, adj != 0), x[i]), y[i]);
    }
}

// constants of the per-wavenumber (L+I)^-1 (App. B.1, forward or conjugated for the adjoint)
struct BaseSymbol {
    float2 P, Pu, c1, c2, c3;  // l1/(a1+l1)/N, l1/(a1+l1), i sqrt(l1 l2), l2 (a1+l1), (a1+l1)(a2+l2)
    float scale;               // 1/N
    const float2* kt[3];       // t_eta
    const float* k2[3];
};

// the per-wavenumber symbol on the C components of each k
template <int C> __global__ void k_base_symbol(Dims d, BaseSymbol Sy, float2* __restrict__ w)
{
    constexpr int D = C - 1;
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < d.N; v += (long long)gridDim.x * blockDim.x) {
        int i0, i1, i2;
        voxel_coords(d, v, i0, i1, i2);
        const int ix[3] = {i0, i1, i2};
        float2 vv[C], t[D], s = make_float2(0.f, 0.f);
        float k2 = 0.f;
#pragma unroll
        for (int c = 0; c < C; ++c) vv[c] = w[c * d.N + v];
#pragma unroll
        for (int e = 0; e < D; ++e) {
            t[e] = Sy.kt[e][ix[e]];
            k2 += Sy.k2[e][ix[e]];
            s = cadd(s, cmulc(vv[e], t[e]));
        }
        const float2 mu = make_float2(k2 + Sy.c3.x, Sy.c3.y);
        const float inv = Sy.scale / cabs2(mu);
        const float2 im = make_float2(mu.x * inv, -mu.y * inv);
        const float2 tmp = cmul(cadd(cmul(Sy.Pu, s), cmul(Sy.c1, vv[D])), im);
#pragma unroll
        for (int e = 0; e < D; ++e) w[e * d.N + v] = csub(cmul(Sy.P, vv[e]), cmul(t[e], tmp));
        w[D * d.N + v] = cmul(csub(cmul(Sy.c2, vv[D]), cmul(Sy.c1, s)), im);
    }
}

// x += nu B (w - x); per-block (|dx|^2, |x|^2) into partials[2 * blockIdx.x]
template <typename R>
__global__ void k_base_update(Dims d, Medium<R> M, cplx<R>* __restrict__ x, const cplx<R>* __restrict__ w, int adj,
                              R nu, double* __restrict__ partials)
{
    const long long n = (long long)(d.D + 1) * d.N;
    R s0 = (R)0, s1 = (R)0;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(i / d.N);
        const long long v = i % d.N;
        int i0, i1, i2;
        voxel_coords(d, v, i0, i1, i2);
        const RowB<R> rb = row_B(M, d.D, c, i1, i2, v - i0);
        const cplx<R> xv = x[i];
        const cplx<R> del = cscale(cmul(born_B(M, rb, i0, adj != 0), csub(w[i], xv)), nu);
        const cplx<R> xn = cadd(xv, del);
        x[i] = xn;
        s0 += cabs2(del);
        s1 += cabs2(xn);
    }
    block_sum2(s0, s1, partials + 2 * (long long)blockIdx.x);
}

}  // namespace cbs
