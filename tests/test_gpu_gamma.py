"""Residuals and steps at other ratios of specific heats than air's, up to far
beyond what the integer flux takes, against the oracle with the parity tests'
bars.  Mach numbers about 1, or 3 / gamma (at more the internal energy is a sliver
that reconstruction noise eats): there too H~ - c~ |u~_n| is negative on many faces."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_2306_14011_gb300 import fv  # noqa: E402
from paper_2306_14011_gb300 import inputs as I  # noqa: E402
from test_gpu_parity import TOL_RES, assert_residual_parity, dev, relerr  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma", [1.1, 5.0 / 3.0, 2.9, 3.2, 5.0, 9.5, 60.0, 1000.0])
@pytest.mark.parametrize("dim", [2, 3])
def test_residual_and_step_match_the_oracle(dim, gamma):
    T = I.BC_TRANSMISSIVE
    g = I.grid2d(61, 75, 1.0, 0.8, T) if dim == 2 else I.grid3d(21, 18, 16, 1.0, 0.9, 0.8)
    W = I.random_smooth(g, seed=4)
    rho, p = W[0], np.sqrt(W[0])
    vel = [2.5 * min(1.0, 3.0 / gamma) * np.sqrt(gamma) * W[1 + d] / rho for d in range(dim)]
    U = I.conserved(rho, tuple(vel), p, gamma)
    so = O.scheme(gamma=gamma)
    dt = O.time_step(g, U, so)
    with fv.Solver(g, gamma=gamma) as s:
        R = s.residual(dev(U)).cpu().numpy()
        V = dev(U)
        s.rk_step(V, dt)
    assert_residual_parity(g, U, R, tag=f"gamma{gamma:g}-{dim}d", s=so)
    assert relerr(V.cpu().numpy(), O.rk3_step(g, U, dt, so)[0]) <= TOL_RES
