"""The scalar form of (L+I)^-1 the kernels run (csrc/born.cuh) and the host side of its dispatch (csrc/launch.cuh), on
the CPU: components merged axis by axis into one sum, solved, and split off again, restated in numpy against the
oracle's entry-by-entry matrix; the row kernels' blocks cover every row of every component once; the padded exchange
layout is a one-to-one, linear map without bank conflicts."""
import ctypes
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

from oracle import oracle as O
from paper_2507_16087_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2507_16087_gb300", "csrc")
SIZES = [8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 512, 1024, 2048]


def scalar_form(v, dx, a1, a2, l1, l2, adjoint, collocated):
    """Axis-by-axis merge, scalar solve and split of (L+I)^-1 v, x first, as the kernels order it."""
    D = v.ndim - 1
    c1, c2, c3, pu = 1j * np.sqrt(l1 * l2), l2 * (a1 + l1), (a1 + l1) * (a2 + l2), l1 / (a1 + l1)
    if adjoint:
        c1, c2, c3, pu = (np.conj(z) for z in (c1, c2, c3, pu))
    t, k2 = [], 0.0
    for e in range(D):
        n = v.shape[D - e]
        k = 2 * np.pi * np.fft.fftfreq(n, dx)
        view = [n if ax == D - 1 - e else 1 for ax in range(D)]
        t.append((k if collocated else k * np.exp(0.5j * k * dx)).reshape(view))
        k2 = k2 + (k ** 2).reshape(view)
    u, q = [v[e].astype(complex) for e in range(D)], v[D].astype(complex)
    for e in range(D):  # forward: transform what is left, merge u_e
        q = np.fft.fft(q, axis=D - 1 - e)
        for f in range(e, D):
            u[f] = np.fft.fft(u[f], axis=D - 1 - e)
        q = q - (c1 / c2) * np.conj(t[e]) * u[e]
    p = c2 * q / (k2 + c3)
    g = [None] * D
    for e in range(D - 1, -1, -1):  # inverse: split the gradient along e, transform what is there
        g[e] = -pu * c1 / (l1 * l2) * t[e] * p
        p = np.fft.ifft(p, axis=D - 1 - e)
        for f in range(e, D):
            g[f] = np.fft.ifft(g[f], axis=D - 1 - e)
    return np.stack([pu * v[e] + g[e] for e in range(D)] + [p])


@pytest.mark.parametrize("shape", [(24, 32), (8, 12), (12, 16, 8), (8, 24, 32)])
@pytest.mark.parametrize("adjoint", [False, True])
@pytest.mark.parametrize("collocated", [False, True])
def test_scalar_form_is_the_inverse_matrix(shape, adjoint, collocated):
    m = W.smooth_random_medium(shape, seed=3, n_abs=2)
    P = O.Problem(m.c0, m.rho, m.alpha, m.dx, m.omega, m.nabs, m.gamma_max, collocated=collocated)
    s = P.scalars()
    v = W.random_source(shape, 5)
    got = scalar_form(v, m.dx, s["a1"], s["a2"], s["lambda1"], s["lambda2"], adjoint, collocated)
    ref = P.green(v, adjoint)
    # the transforms' rounding, eps log N, times a few
    assert np.linalg.norm(got - ref) <= 1e-13 * np.linalg.norm(ref)


SRC = r'''
#include "launch.cuh"
using namespace cbs;

// every (component, row) a row block's units address, as k_rows decodes its block: hits[c * rows + row] += 1
template <typename R, int N> int cover(int D, int n1, int n2, int* hits, int* threads) {
    Dims d; d.D = D; d.n0 = N; d.n1 = n1; d.n2 = n2; d.N = (long long)N * n1 * n2;
    const RowGrid g = row_grid<R, N>(d);
    const int rx = rows_tiny<R, N>(d) ? r_rows_tile<R>(N) : r_rows<R>(N);
    *threads = g.units * (N / rx);
    const long long rpc = d.N / N;
    const int U = g.units, H = U / 2;
    for (int blk = 0; blk < g.blocks; ++blk) {
        const bool pair = blk < g.npair;
        const int per = pair ? H : U;
        int c = pair ? D : 1 + (blk - g.npair) / g.nsingle, b = pair ? blk : (blk - g.npair) % g.nsingle;
        for (int lu = 0; lu < U; ++lu) {
            const bool isx = pair && lu >= H;
            const long long row = (long long)b * per + (isx ? lu - H : lu);
            if (row < rpc && (row - (long long)b * per) < per) hits[(isx ? 0 : c) * rpc + row] += 1;
        }
    }
    return g.blocks;
}
extern "C" int rows_cover(int f64, int D, int n0, int n1, int n2, int* hits, int* threads) {
    switch (n0) {
#define CBS_CASE(N) case N: return f64 ? cover<double, N>(D, n1, n2, hits, threads) : cover<float, N>(D, n1, n2, hits, threads);
        CBS_FOR_EACH_SIZE(CBS_CASE)
#undef CBS_CASE
    }
    return -1;
}

// padded positions of a row in the split the exchange uses: pos[j * parts + k] for thread part j, compile-time part k
template <typename CT, int N, int T, int K = 0> void layout_k(int stride, int* pos) {
    if constexpr (K * 2 < N) {
        for (int j = 0; j < N / 2; ++j) { pos[2 * j] = RowPad<CT, N, T>::at(j, 0); pos[2 * j + 1] = RowPad<CT, N, T>::at(j, N / 2); }
    }
}
template <typename R, int N> int pitch(int* pos) {
    using CT = cplx<R>;
    constexpr int T = N / r_rows<R>(N);
    layout_k<CT, N, T>(N / 2, pos);
    return RowPad<CT, N, T>::SL;
}
extern "C" int row_pitch(int f64, int n, int* pos) {
    switch (n) {
#define CBS_CASE(N) case N: return f64 ? pitch<double, N>(pos) : pitch<float, N>(pos);
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
    src, so = os.path.join(d, "rows.cu"), os.path.join(d, "rows.so")
    open(src, "w").write(SRC)
    subprocess.check_call([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-Xcompiler", "-fPIC",
                           "-shared", "-I" + CSRC, "-I" + os.path.join(ROOT, "include"), src, "-o", so])
    L = ctypes.CDLL(so)
    L.rows_cover.argtypes = [ctypes.c_int] * 5 + [ctypes.c_void_p] * 2
    L.row_pitch.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_void_p]
    return L


@pytest.mark.parametrize("f64", [0, 1])
@pytest.mark.parametrize("n0", SIZES)
@pytest.mark.parametrize("rest", [(2, 8, 1), (2, 192, 1), (3, 12, 8), (3, 24, 48)])
def test_row_blocks_cover_every_row_once(lib, f64, n0, rest):
    D, n1, n2 = rest
    hits = np.zeros((D + 1) * n1 * n2, dtype=np.int32)
    threads = ctypes.c_int()
    assert lib.rows_cover(f64, D, n0, n1, n2, hits.ctypes.data, ctypes.byref(threads)) > 0
    assert hits.min() == hits.max() == 1
    assert threads.value % 32 == 0 and threads.value <= 1024


@pytest.mark.parametrize("f64", [0, 1])
@pytest.mark.parametrize("n", SIZES)
def test_padded_rows_are_one_to_one(lib, f64, n):
    pos = np.full(n, -1, dtype=np.int32)
    sl = lib.row_pitch(f64, n, pos.ctypes.data)
    order = np.empty(n, dtype=np.int64)  # position of element e, in the order the split gave them
    order[: n // 2], order[n // 2:] = pos[0::2], pos[1::2]
    sh = 3 if f64 else 4
    e = np.arange(n)
    assert np.array_equal(order, e + (e >> sh))     # the split map is the map itself
    assert order.max() < sl and len(set(order)) == n
    assert (sl * (16 if f64 else 8)) % 16 == 0      # rows start where a bulk copy may
