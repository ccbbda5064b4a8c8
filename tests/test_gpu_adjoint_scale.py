"""The VJPs are linear in the cotangent: scaled by a power of two, down to where
the residual's VJP is a few hundred times the smallest normal number, it gives
the scaled result.

Tolerance: the terms of one scale are rounded once more in the other (an
operation may round in FP64 where the integer pipes keep more), 1e-12 of the
largest result as in the adjoint's tests, and a subnormal number's spacing for
each of some thousand operations."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2306_14011_gb300 import fv  # noqa: E402
from paper_2306_14011_gb300 import inputs as I  # noqa: E402
from test_gpu_adjoint import dev  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exponent", [900, 400, -490, -510, -900, -990, -1010])
@pytest.mark.parametrize("dim", [2, 3])
def test_the_vjp_scales_with_the_cotangent(dim, exponent):
    g = I.grid2d(37, 26, 1.0, 0.7, ((1, 1), (0, 0), (0, 0))) if dim == 2 else I.grid3d(11, 9, 10, 1.0, 0.7, 0.8)
    U = dev(I.random_smooth(g, seed=dim))
    lam = np.random.default_rng(3).normal(size=g.shape)
    lam[:, ..., 3:7] = 0.0  # no cotangent in a part of the grid
    with fv.Solver(g) as s:
        dt = s.time_step(U)
        for vjp in (s.residual_vjp, lambda U, l: s.rk_step_vjp(U, l, dt)):
            ref = vjp(U, dev(lam)).cpu().numpy()
            got = np.ldexp(vjp(U, dev(np.ldexp(lam, exponent))).cpu().numpy(), -exponent)
            assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max() + 1e4 * 2.0 ** (-1074 - exponent)
