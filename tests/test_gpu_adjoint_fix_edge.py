"""The residual's VJP at faces next to the edge of the entropy fix, |u~_n - c~| =
delta (1 +- eps) with eps from 2^-20 to 2^-40, on either side and for either sign.
The flux has a continuous slope there and a jump in its curvature, so the wrong
branch is off by eps / 2 times a wave strength (decided in FP32: 1e-11 of the result).
Two constant states meet at one face (the limiter's slopes are zero, so they are
the face's states), with the velocity that puts the face there.  Against the
Jacobian of the oracle's dual numbers, with the bar of the adjoint's tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_2306_14011_gb300 import fv  # noqa: E402
from paper_2306_14011_gb300 import inputs as I  # noqa: E402
from test_gpu_adjoint import _full_jacobian_T_lam, dev  # noqa: E402

pytestmark = pytest.mark.gpu

EFIX = 0.1


def edge_state(g, rng, where):
    """Cells of a random left and right state whose face has u~_x - c~ = where c~."""
    rho, p, u, v = rng.uniform(0.8, 1.3, 2), rng.uniform(0.8, 1.3, 2), rng.uniform(-0.2, 0.2, 2), rng.uniform(-0.3, 0.3, 2)
    w = np.sqrt(rho) / np.sqrt(rho).sum()
    for _ in range(30):  # a common velocity: c~ does not depend on it but for rounding
        H = 1.4 / 0.4 * p / rho + 0.5 * (u * u + v * v)
        un = (w * u).sum()
        c = np.sqrt(0.4 * ((w * H).sum() - 0.5 * (un ** 2 + (w * v).sum() ** 2)))
        u = u + (c * (1.0 + where) - un)
    side = (np.arange(g.n[0]) >= g.n[0] // 2).astype(int)
    one = np.ones(g.shape[1:])
    return I.conserved(rho[side] * one, (u[side] * one, v[side] * one), p[side] * one)


@pytest.mark.parametrize("bits", [20, 22, 23, 24, 26, 30, 40])
@pytest.mark.parametrize("edge", [-1, 1])
def test_vjp_at_the_edge_of_the_fix(edge, bits):
    g = I.grid2d(6, 2, 1.0, 0.4, ((1, 1), (0, 0), (0, 0)))
    rng = np.random.default_rng(bits)
    with fv.Solver(g, efix=EFIX) as s:
        for side in (-1, 1, -1, 1, -1, 1):
            U = edge_state(g, rng, edge * EFIX * (1.0 + side * 2.0 ** -bits))
            lam = rng.normal(size=U.shape)
            ref = _full_jacobian_T_lam(g, U, lam)
            got = s.residual_vjp(dev(U), dev(lam)).cpu().numpy()
            assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
