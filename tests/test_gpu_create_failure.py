"""solver_create when the caller's allocator runs out at each of its allocations in turn, also while the host-made tables
are still being copied: CBS_ENOMEM, everything given back, and the solver made next is right."""

import numpy as np
import pytest

from oracle import oracle as O
from paper_2507_16087_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_allocation_failures_give_everything_back(precision, monkeypatch):
    from paper_2507_16087_gb300 import cbs

    shape = (24, 32)
    p = W.smooth_random_medium(shape, seed=65, n_abs=2)
    T = lambda a: torch.tensor(np.ascontiguousarray(a), device=DEV)  # noqa: E731
    args = (T(p.c0), T(p.rho), T(p.alpha), p.dx, p.omega, p.nabs, p.gamma_max)
    live, left = set(), [0]

    def allocator(stream):
        def alloc(nbytes, _stream, _ctx):
            if left[0] == 0:
                return None
            left[0] -= 1
            ptr = torch.cuda.caching_allocator_alloc(int(nbytes), device=stream.device, stream=stream)
            live.add(ptr)
            return ptr

        def free(ptr, _ctx):
            live.remove(ptr)
            torch.cuda.caching_allocator_delete(ptr)

        return cbs.DEV_ALLOC_FN(alloc), cbs.DEV_FREE_FN(free)

    monkeypatch.setattr(cbs, "_torch_allocator", allocator)
    for k in range(200):
        left[0] = k
        try:
            s = cbs.solver_create(*args, precision=precision, allocator="torch", tol=0.0, max_iter=10, nu=0.5)
            break
        except cbs.CBSError as e:
            assert e.status == cbs.CBS_ENOMEM
            assert not live
    else:
        pytest.fail("the solver needs more allocations than it was given")
    assert k > 10
    src = W.random_source(shape, 66)
    out = torch.empty(s.field_shape, dtype=torch.complex128, device=DEV)
    s.solve_forward(T(src), out)
    P = O.Problem(p.c0, p.rho, p.alpha, p.dx, p.omega, p.nabs, p.gamma_max)
    x, _ = P.iterate(P.scale_source(src), n_iter=10, nu=0.5)
    ref = P.unscale(x)
    assert np.linalg.norm(out.cpu().numpy() - ref) <= (1e-11 if precision == "fp64" else 1e-5) * np.linalg.norm(ref)
    s.destroy()
    assert not live
