"""The scalar-form kernels at the edges of their tiles and of their dispatch, against the FP64 oracle: row blocks with
fewer rows than units, columns that do not fill a tile, halves of the u_z columns that do not, grids on either side of
the small-tile and few-values rules, rows whose y goes straight to registers; solves of a fixed number of iterations
(the update kernel without norms), a warm start, and applies in place.

Tolerances as in test_gpu_parity.py: one apply 1e-12 (float64) and 2e-6 (float32), 20 iterations 1e-11 and 1e-5."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2507_16087_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
# (n1, n0) or (n2, n1, n0)
SHAPES = [(8, 8), (12, 12), (8, 2048), (24, 1024), (512, 24), (1024, 12), (8, 8, 8), (8, 12, 24), (12, 8, 12),
          (16, 192, 16), (96, 96, 8), (8, 64, 96), (64, 16, 64), (32, 32, 32)]


def T(a):
    return torch.tensor(np.ascontiguousarray(a), device=DEV)


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def make(shape, precision, seed=60, **kw):
    from paper_2507_16087_gb300 import cbs

    p = W.smooth_random_medium(shape, seed=seed, n_abs=2)
    p.gamma_max = 0.5 * p.omega
    s = cbs.solver_create(T(p.c0), T(p.rho), T(p.alpha), p.dx, p.omega, p.nabs, p.gamma_max, precision=precision, nu=0.5, **kw)
    return s, O.Problem(p.c0, p.rho, p.alpha, p.dx, p.omega, p.nabs, p.gamma_max)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("precision,tol1,tol20", [("fp64", 1e-12, 1e-11), ("fp32", 2e-6, 1e-5)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_applies_and_fixed_iterations_match_oracle(shape, precision, tol1, tol20, adjoint):
    s, P = make(shape, precision, tol=0.0, max_iter=20)
    v = W.random_source(shape, 61)
    out = torch.full(s.field_shape, complex(np.nan, np.nan), dtype=torch.complex128, device=DEV)
    s.green_apply(T(v), out, adjoint)
    assert rel(out.cpu().numpy(), P.green(v, adjoint)) <= tol1
    s.operator_apply(T(v), out, adjoint)
    assert rel(out.cpu().numpy(), P.apply(v, adjoint)) <= 1e-12
    (s.solve_adjoint if adjoint else s.solve_forward)(T(v), out)
    x, _ = P.iterate(P.scale_source(v, adjoint), n_iter=20, nu=0.5, adjoint=adjoint)
    assert rel(out.cpu().numpy(), P.unscale(x)) <= tol20
    # a warm start goes on from there
    (s.solve_adjoint if adjoint else s.solve_forward)(T(v), out, x0=out.clone())
    x, _ = P.iterate(P.scale_source(v, adjoint), n_iter=40, nu=0.5, adjoint=adjoint)
    assert rel(out.cpu().numpy(), P.unscale(x)) <= 2 * tol20


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_applies_in_place_and_partly_overlapping(precision):
    """in == out, and an output that starts inside the input, give what separate buffers give."""
    shape = (12, 16, 24)
    s, _ = make(shape, precision)
    n = int(np.prod(s.field_shape))
    v = T(W.random_source(shape, 62))
    for fn in (s.green_apply, s.operator_apply):
        ref = torch.empty_like(v)
        fn(v, ref)
        same = v.clone()
        fn(same, same)
        assert torch.equal(same, ref)
        buf = torch.empty(n + 8, dtype=torch.complex128, device=DEV)
        a, b = buf[:n].view(s.field_shape), buf[8:].view(s.field_shape)
        a.copy_(v)
        fn(a, b)
        assert torch.equal(b, ref)
