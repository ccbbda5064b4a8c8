"""Long van Leer runs of rotated Sod problems.  Ahead of the front the momenta
decay through the subnormal range while the rest of the state stays near 1, so
the limiter meets subnormal differences inside a normal state; with a reciprocal
that flushes them a slope there is NaN and spreads over the grid.  States against
the oracle, with the 100-step bar of the parity tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_2306_14011_gb300 import fv  # noqa: E402
from paper_2306_14011_gb300 import inputs as I  # noqa: E402
from test_gpu_parity import TOL_100, dev, relerr  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("recon", [fv.FV_RECON_CONSERVED, fv.FV_RECON_PRIMITIVE])
@pytest.mark.parametrize("theta", [0.35, 1.9, 2.6, 4.1, 5.5])
def test_a_hundred_steps_stay_finite_and_match_the_oracle(theta, recon):
    g, U = I.sod_rotated(100, theta)
    with fv.Solver(g, limiter=fv.FV_LIM_VANLEER, recon=recon) as s:
        Ud = dev(U)
        t = s.run(Ud, 100, return_time=True)
    U100 = Ud.cpu().numpy()
    Uo, to = O.run(g, U, 100, s=O.scheme(limiter=O.LIM_VANLEER, recon=recon))
    assert np.isfinite(Uo).all() and np.isfinite(U100).all()
    assert relerr(U100, Uo) <= TOL_100
    assert abs(t - to) <= 1e-12 * to
