"""2D grids of few 2048-point rows, whose rows run a block each (u_x's too, merged and split at the last axis), and the first
grid above that rule, against the FP64 oracle: applies, iterations with and without their increments, residual, both grids.

Tolerances as in test_gpu_parity.py: one apply 1e-12 (float64) and 2e-6 (float32), 20 iterations 1e-11 and 1e-5, increments
1e-9 and 1e-4."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2507_16087_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def T(a):
    return torch.tensor(np.ascontiguousarray(a), device=DEV)


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("n1,collocated", [(8, False), (12, True), (24, False), (48, False), (64, False)])
@pytest.mark.parametrize("precision,tol1,tol20,tolinc", [("fp64", 1e-12, 1e-11, 1e-9), ("fp32", 2e-6, 1e-5, 1e-4)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_few_long_rows_match_oracle(n1, collocated, precision, tol1, tol20, tolinc, adjoint):
    from paper_2507_16087_gb300 import cbs

    shape = (n1, 2048)
    p = W.smooth_random_medium(shape, seed=80, n_abs=2)
    p.gamma_max = 0.5 * p.omega
    s = cbs.solver_create(T(p.c0), T(p.rho), T(p.alpha), p.dx, p.omega, p.nabs, p.gamma_max, precision=precision, nu=0.5,
                          tol=0.0, max_iter=20, check_every=8, collocated=collocated)
    P = O.Problem(p.c0, p.rho, p.alpha, p.dx, p.omega, p.nabs, p.gamma_max, collocated=collocated)
    v = W.random_source(shape, 81)
    out = torch.full(s.field_shape, complex(np.nan, np.nan), dtype=torch.complex128, device=DEV)
    s.green_apply(T(v), out, adjoint)
    assert rel(out.cpu().numpy(), P.green(v, adjoint)) <= tol1
    s.operator_apply(T(v), out, adjoint)
    assert rel(out.cpu().numpy(), P.apply(v, adjoint)) <= 1e-12
    y = P.scale_source(v, adjoint)
    x, inc = P.iterate(y, n_iter=20, nu=0.5, adjoint=adjoint)
    (s.solve_adjoint if adjoint else s.solve_forward)(T(v), out)
    assert rel(out.cpu().numpy(), P.unscale(x)) <= tol20
    xg = torch.zeros_like(out)
    got = s.born_iterate(T(y), xg, 20, adjoint)
    assert rel(xg.cpu().numpy(), x) <= tol20
    assert np.max(np.abs(got - inc) / inc) <= tolinc
    r = y - P.apply(x, adjoint)
    assert abs(s.residual_norm(T(P.unscale(x)), T(v), adjoint) - np.linalg.norm(r) / np.linalg.norm(y)) <= 1e-10
