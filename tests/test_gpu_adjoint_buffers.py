"""The adjoint's work states outlive a residual that grows the norm buffer."""
import pytest

torch = pytest.importorskip("torch")

from paper_2306_14011_gb300 import fv  # noqa: E402
from paper_2306_14011_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


def test_step_vjp_after_a_residual_with_norms():
    g, U0 = I.isentropic_vortex(96, seed=0)
    U = torch.from_numpy(U0).cuda()
    lam = torch.randn_like(U)
    with fv.Solver(g) as s:
        dt = s.time_step(U)
        before = s.rk_step_vjp(U, lam, dt)
        s.residual(U, norms=True)  # allocates the norm partials on this first call
        other = [torch.full_like(U, float("nan")) for _ in range(8)]  # takes up memory that had been given back
        assert torch.equal(s.rk_step_vjp(U, lam, dt), before)
        del other
