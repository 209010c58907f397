"""The scaled source where it is formed (scale_source, and inside a float32 solve), against the FP64 oracle: dense sources,
sources with zeros among the values and whole zero components, one value a thread and several with an odd one left over.

Tolerances as in test_gpu_parity.py: the scaling alone 1e-14, one float32 iteration 1e-5."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2507_16087_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def T(a):
    return torch.tensor(np.ascontiguousarray(a), device=DEV)


def sources(shape):
    dense = W.random_source(shape, 71)
    rng = np.random.default_rng(72)
    mixed = dense * (rng.random(dense.shape) < 0.3)
    mixed[0] = 0.0
    mixed.real[1] *= rng.random(shape) < 0.5  # one part zero is not a zero value
    point = np.zeros_like(dense)
    point[(len(shape),) + tuple(n // 2 for n in shape)] = 1.0 - 2.0j
    return {"dense": dense, "mixed": mixed, "point": point}


@pytest.mark.parametrize("shape", [(8, 8), (24, 32), (12, 16, 24), (96, 128, 128)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_scaled_source_matches_oracle(shape, adjoint):
    from paper_2507_16087_gb300 import cbs

    p = W.smooth_random_medium(shape, seed=70, n_abs=2)
    P = O.Problem(p.c0, p.rho, p.alpha, p.dx, p.omega, p.nabs, p.gamma_max)
    s = cbs.solver_create(T(p.c0), T(p.rho), T(p.alpha), p.dx, p.omega, p.nabs, p.gamma_max, precision="fp32", nu=0.5,
                          tol=0.0, max_iter=1)
    out = torch.empty(s.field_shape, dtype=torch.complex128, device=DEV)
    for name, src in sources(shape).items():
        y = P.scale_source(src, adjoint)
        out.fill_(complex(np.nan, np.nan))
        s.scale_source(T(src), out, adjoint)
        got = out.cpu().numpy()
        assert np.linalg.norm(got - y) <= 1e-14 * np.linalg.norm(y), name
        assert np.array_equal(got == 0, y == 0), name
        out.fill_(complex(np.nan, np.nan))
        (s.solve_adjoint if adjoint else s.solve_forward)(T(src), out)
        x, _ = P.iterate(y, n_iter=1, nu=0.5, adjoint=adjoint)
        ref = P.unscale(x)
        assert np.linalg.norm(out.cpu().numpy() - ref) <= 1e-5 * np.linalg.norm(ref), name
