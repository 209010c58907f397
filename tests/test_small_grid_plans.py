"""FFT plans of the values-per-thread counts that only the small-grid rules choose (csrc/launch.cuh: r_tile, r_rows_tile),
checked on the host: the radices multiply to the length and divide the thread's count, every pass's slot order is a
permutation with q_slot its inverse, and the padded exchange's split into a thread's part and a compile-time part is the
padding of their sum at every offset that a pass uses."""
import ctypes
import os
import shutil
import subprocess
import tempfile

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2507_16087_gb300", "csrc")
SIZES = [8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 512, 1024, 2048]

SRC = r'''
#include "launch.cuh"
using namespace cbs;

template <typename CT, int N, int R, int P> int pass_ok()
{
    constexpr int np = plan_npass(N, R);
    if constexpr (P <= np) {
        bool seen[R] = {};
        for (int s = 0; s < R; ++s) {
            const int q = slot_q<N, R, P>(s);
            if (q < 0 || q >= R || seen[q] || q_slot<N, R, P>(q) != s) return 10 + P;
            seen[q] = true;
        }
        if constexpr (P + 1 < np) {  // the exchange after pass P: writes, then reads in pass P + 1's order
            using L = RowPad<CT, N, N / R>;
            constexpr int T = N / R, r = plan_radix(N, R, P), ns = plan_ns(N, R, P), rn = plan_radix(N, R, P + 1);
            for (int j = 0; j < N / r; ++j)
                for (int k = 0; k < r; ++k) {
                    const int idx = (j / ns) * ns * r + j % ns;
                    if (L::at(idx, k * ns) != L::pad(idx + k * ns)) return 30 + P;
                }
            for (int t = 0; t < T; ++t)
                for (int m = 0; m < R / rn; ++m)
                    for (int k = 0; k < rn; ++k)
                        if (L::at(t + T * m, k * (N / rn)) != L::pad(t + T * m + k * (N / rn))) return 50 + P;
        }
        return pass_ok<CT, N, R, P + 1>();
    }
    return 0;
}
template <typename R, int N, int V> int plan_ok()
{
    constexpr int np = plan_npass(N, V);
    if (np <= 0 || N % V != 0) return 1;
    int prod = 1;
    for (int p = 0; p < np; ++p) {
        const int r = plan_radix(N, V, p);
        if (V % r != 0) return 2;
        prod *= r;
    }
    if (prod != N) return 3;
    return pass_ok<cplx<R>, N, V, 0>();
}
extern "C" int check(int n, int which)
{
    switch (n) {
#define CBS_CASE(N) case N: return which == 0 ? plan_ok<double, N, r_tile<double>(N)>() : which == 1 ? plan_ok<float, N, r_rows_tile<float>(N)>() \
                                                                                             : plan_ok<float, N, r_tile<float>(N)>();
        CBS_FOR_EACH_SIZE(CBS_CASE)
#undef CBS_CASE
    }
    return -1;
}
'''


@pytest.fixture(scope="module")
def lib():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = tempfile.mkdtemp()
    src, so = os.path.join(d, "small.cu"), os.path.join(d, "small.so")
    open(src, "w").write(SRC)
    subprocess.check_call([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-Xcompiler", "-fPIC",
                           "-shared", "-I" + CSRC, "-I" + os.path.join(ROOT, "include"), src, "-o", so])
    L = ctypes.CDLL(so)
    L.check.argtypes = [ctypes.c_int, ctypes.c_int]
    return L


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("which", [0, 1, 2])  # float64 tiles and rows, float32 rows, float32 tiles
def test_small_grid_plans(lib, n, which):
    assert lib.check(n, which) == 0
