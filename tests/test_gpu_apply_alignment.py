"""The float64 applies on buffers that lie on 8 bytes only (C's alignment of double complex), called through the C ABI:
the same values as on aligned buffers, and nothing written outside the output."""
import ctypes

import numpy as np
import pytest

from paper_2507_16087_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("shape", [(24, 32), (12, 16, 24)])
@pytest.mark.parametrize("name", ["green_apply", "operator_apply"])
@pytest.mark.parametrize("off_in,off_out", [(1, 0), (0, 1), (1, 1)])
def test_applies_take_buffers_on_eight_bytes(shape, name, off_in, off_out):
    from paper_2507_16087_gb300 import cbs

    p = W.smooth_random_medium(shape, seed=63, n_abs=2)
    T = lambda a: torch.tensor(np.ascontiguousarray(a), device=DEV)  # noqa: E731
    s = cbs.solver_create(T(p.c0), T(p.rho), T(p.alpha), p.dx, p.omega, p.nabs, p.gamma_max, precision="fp64")
    v = T(W.random_source(shape, 64))
    ref = torch.empty_like(v)
    getattr(s, name)(v, ref)
    n = 2 * v.numel()
    src = torch.empty(n + 2, dtype=torch.float64, device=DEV)
    dst = torch.full((n + 4,), 7.0, dtype=torch.float64, device=DEV)
    src[off_in:off_in + n] = torch.view_as_real(v).reshape(-1)
    at = 2 + off_out  # guard values on both sides
    fn = getattr(cbs.load(), name)
    call = lambda a, b: fn(s._h, ctypes.c_void_p(a), ctypes.c_void_p(b), 0)  # noqa: E731
    torch.cuda.synchronize()
    assert call(src.data_ptr() + 8 * off_in, dst.data_ptr() + 8 * at) == cbs.CBS_OK
    assert torch.equal(dst[at:at + n], torch.view_as_real(ref).reshape(-1))
    assert bool((dst[:at] == 7.0).all()) and bool((dst[at + n:] == 7.0).all())
    # in place, off the boundary
    if off_in and off_out:
        a = src.data_ptr() + 8 * off_in
        assert call(a, a) == cbs.CBS_OK
        assert torch.equal(src[off_in:off_in + n], torch.view_as_real(ref).reshape(-1))
