"""Launches of the kernels of an iteration (csrc/launch.cuh), on the CPU: the launchers run against a stand-in for the
runtime's launch call that records each launch.  A row block must not take shared memory that its mode or row length
never touches, or fewer blocks fit on an SM than the kernel was compiled for; a strided axis takes its small tile only
where that makes more blocks."""
import ctypes
import os
import shutil
import subprocess
import tempfile

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2507_16087_gb300", "csrc")
FWD, FUSED, FUSED_NORM, INV, COPY, GREEN = range(6)  # RowsMode

SRC = r'''
#include <cuda_runtime.h>
static int g_threads, g_smem, g_blocks, g_early, g_early_arg;
extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void** args)
{
    g_threads = c->blockDim.x; g_smem = (int)c->dynamicSmemBytes; g_blocks = c->gridDim.x;
    if (g_early_arg > 0) g_early = *(const int*)args[g_early_arg];
    return cudaSuccess;
}
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
#include "launch.cuh"
using namespace cbs;
using P32 = Plan<float>;

template <typename R, int N> int run(int D, int n1, int n2, int mode, int* o)
{
    Plan<R> P{};
    P.d.D = D; P.d.n0 = N; P.d.n1 = n1; P.d.n2 = n2; P.d.N = (long long)N * n1 * n2;
    const bool tiny = rows_tiny<R, N>(P.d);
    const cudaError_t e = rows_n<R, N>(P, nullptr, nullptr, nullptr, mode, 0, (R)0, nullptr, nullptr);
    using A = RowCfg<R, N, r_rows<R>(N)>;
    using B = RowCfg<R, N, r_rows_tile<R>(N)>;
    o[0] = g_threads; o[1] = g_smem; o[2] = g_blocks;
    o[3] = tiny ? B::MINB : A::MINB;                       // blocks an SM the kernel is compiled for
    o[4] = (tiny ? B::SL : A::SL) * (int)sizeof(cplx<R>);  // a field row
    o[5] = (tiny ? B::ML : A::ML) * (int)sizeof(R);        // a medium row
    o[6] = g_threads / (tiny ? B::T : A::T);               // units
    return (int)e;
}
// whether a float32 axis of N points and `columns` columns takes the small tile, and the blocks either tile makes
template <int N> int tiles(long long columns, int* o)
{
    P32 P{};
    P.d.D = 2; P.d.n0 = (int)columns; P.d.n1 = N; P.d.n2 = 1; P.d.N = columns * N;
    const cudaError_t e = last2_n<float, N>(P, nullptr, 0, nullptr);
    o[0] = g_blocks; o[1] = g_threads;
    o[2] = (int)((columns + cols_big<float>(N) - 1) / cols_big<float>(N));
    o[3] = N / r_axis<float>(N) * cols_big<float>(N);
    return (int)e;
}
// the early flags of the row and the last-axis kernel of a 2D grid (arguments 10 of k_rows, 4 of k_last2)
template <int N0, int N1> int early2(int* o)
{
    P32 P{};
    P.d.D = 2; P.d.n0 = N0; P.d.n1 = N1; P.d.n2 = 1; P.d.N = (long long)N0 * N1;
    g_early_arg = 10;
    cudaError_t e = rows_n<float, N0>(P, nullptr, nullptr, nullptr, ROWS_FUSED, 0, 0.0f, nullptr, nullptr);
    o[0] = g_early;
    g_early_arg = 4;
    if (e == cudaSuccess) e = last2_n<float, N1>(P, nullptr, 0, nullptr);
    o[1] = g_early;
    g_early_arg = 0;
    return (int)e;
}
extern "C" int early(int k, int* o)
{
    switch (k) {
    case 0: return early2<2048, 24>(o);
    case 1: return early2<2048, 96>(o);
    case 2: return early2<512, 192>(o);
    case 3: return early2<128, 128>(o);
    case 4: return early2<1024, 1024>(o);
    }
    return -1;
}
extern "C" int last_launch(int n, long long columns, int* o)
{
    switch (n) {
    case 64: return tiles<64>(columns, o);
    case 512: return tiles<512>(columns, o);
    case 1024: return tiles<1024>(columns, o);
    case 2048: return tiles<2048>(columns, o);
    }
    return -1;
}
extern "C" int row_launch(int f64, int D, int n0, int n1, int n2, int mode, int* o)
{
    if (!f64 && n0 == 2048) return run<float, 2048>(D, n1, n2, mode, o);
    if (!f64 && n0 == 1024) return run<float, 1024>(D, n1, n2, mode, o);
    if (!f64 && n0 == 64) return run<float, 64>(D, n1, n2, mode, o);
    if (f64 && n0 == 64) return run<double, 64>(D, n1, n2, mode, o);
    return -1;
}
'''


@pytest.fixture(scope="module")
def lib():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = tempfile.mkdtemp()
    src, so = os.path.join(d, "mem.cu"), os.path.join(d, "mem.so")
    open(src, "w").write(SRC)
    # PTX only (nothing here runs on a device); the shared runtime and references bound within the library, so that the
    # stand-ins above take the place of its calls
    subprocess.check_call([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=compute_103a", "-cudart", "shared",
                           "-Xlinker", "-Bsymbolic", "-Xcompiler", "-fPIC", "-shared", "-I" + CSRC, "-I" + os.path.join(ROOT, "include"), src,
                           "-o", so])
    L = ctypes.CDLL(so)
    L.row_launch.argtypes = [ctypes.c_int] * 6 + [ctypes.c_void_p]
    L.last_launch.argtypes = [ctypes.c_int, ctypes.c_longlong, ctypes.c_void_p]
    L.early.argtypes = [ctypes.c_int, ctypes.c_void_p]
    return L


def launched(lib, f64, grid, mode):
    D = len(grid)
    o = (ctypes.c_int * 7)()
    assert lib.row_launch(f64, D, grid[0], grid[1], grid[2] if D == 3 else 1, mode, o) == 0
    return dict(zip(("threads", "smem", "blocks", "minb", "row", "mrow", "units"), o))


@pytest.mark.parametrize("grid", [(2048, 64), (2048, 512), (2048, 2048), (1024, 12), (1024, 512), (1024, 1024),
                                  (1024, 8, 16), (2048, 8, 8)])
@pytest.mark.parametrize("mode", [FWD, FUSED, FUSED_NORM, INV])
def test_long_rows_fit_the_blocks_an_sm_they_are_compiled_for(lib, grid, mode):
    g = launched(lib, 0, grid, mode)
    assert g["minb"] >= 2
    # 228 KiB of shared memory an SM; 1 KiB of it and the norms' 512 B of static scratch go with each block
    assert g["minb"] * (g["smem"] + 1024 + 512) <= 228 * 1024


@pytest.mark.parametrize("f64,grid", [(0, (2048, 64)), (0, (1024, 2048)), (0, (64, 12)), (0, (64, 64, 64)), (1, (64, 12)),
                                      (1, (64, 64, 64))])
@pytest.mark.parametrize("mode", range(6))
def test_a_launch_asks_for_the_buffers_its_mode_uses(lib, f64, grid, mode):
    g = launched(lib, f64, grid, mode)
    fields = 1 if mode in (COPY, GREEN) else 2  # x and w; only the exchange in the modes without B
    medium = 0 if mode in (COPY, GREEN) else g["units"] // 2 * 3 * g["mrow"]
    least = g["units"] * fields * g["row"] + medium
    # y may have a buffer of its own in the updates, for rows whose y is staged; the barriers take up to 32 bytes
    own_y = g["units"] * g["row"] if mode in (FUSED, FUSED_NORM, INV) and not (grid[0] >= 1024 and not f64) else 0
    assert g["smem"] in (least, least + 32, least + own_y + 32)


@pytest.mark.parametrize("n", [64, 512, 1024, 2048])
@pytest.mark.parametrize("columns", [8, 48, 128, 512, 1024, 2048])
def test_a_small_tile_is_taken_for_more_blocks(lib, n, columns):
    o = (ctypes.c_int * 4)()
    assert lib.last_launch(n, columns, o) == 0
    blocks, threads, big_blocks, big_threads = o
    assert (blocks, threads) == (big_blocks, big_threads) or (blocks > big_blocks and threads <= big_threads)


# 2048 x 24: 36 row blocks before 128 warps, 128 last-axis blocks before 288; 2048 x 96: 144 row blocks before 512 warps, 512
# last-axis blocks; 512 x 192: the last axis before 1152 warps of rows; 128^2: 192 row blocks, the last axis before 192
# warps; 1024^2: more than a block an SM everywhere
@pytest.mark.parametrize("case,rows,last", [(0, 1, 1), (1, 0, 0), (2, 0, 0), (3, 0, 1), (4, 0, 0)])
def test_the_next_kernel_starts_early_where_it_does_not_crowd(lib, case, rows, last):
    o = (ctypes.c_int * 2)()
    assert lib.early(case, o) == 0
    assert list(o) == [rows, last]
