"""The van Leer slope on the integer pipes: states scaled by powers of two, down
to where its operands (and the flux's) go to FP64.  The limiter and the flux are
homogeneous of degree one, so the residual scales exactly; two evaluations of
it differ by at most the 8 ulps of the summed terms of the parity tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_2306_14011_gb300 import fv  # noqa: E402
from paper_2306_14011_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [-980, -600, -280, 0, 280, 900])
@pytest.mark.parametrize("dim", [2, 3])
def test_the_residual_scales_with_the_state(dim, exponent):
    T = I.BC_TRANSMISSIVE
    g = I.grid2d(53, 41, 1.0, 1.0, T) if dim == 2 else I.grid3d(17, 13, 11, 1.0, 1.0, 1.0, T)
    U = I.random_smooth(g, seed=2)
    U[:, ..., 5:9] = U[:, ..., 5:6]  # equal neighbours: zero differences
    s = O.scheme(limiter=1)
    ref = O.residual(g, U, s)
    tol = 8 * np.finfo(float).eps * O.residual_terms(g, U, s).reshape(g.nvar, -1).max(axis=1)
    with fv.Solver(g, limiter=fv.FV_LIM_VANLEER) as sol:
        R = sol.residual(torch.from_numpy(U * 2.0 ** exponent).cuda()).cpu().numpy() * 2.0 ** -exponent
    assert np.all(np.abs(R - ref).reshape(g.nvar, -1).max(axis=1) <= tol)
