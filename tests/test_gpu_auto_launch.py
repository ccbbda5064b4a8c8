"""The launch a context takes when it is given none: the tiles change with the
grid (auto_launch in fv_api.cu), the results do not.  Grids on both sides of
each change of tile on a 152-SM GPU (608 CTAs of one tile shape), odd and even
widths, ragged tiles, and on both sides of the one-pass time-step reduction
(65536 cells).  Equality is exact, so there is no tolerance to choose."""
import pytest

torch = pytest.importorskip("torch")

from paper_2306_14011_gb300 import fv  # noqa: E402
from paper_2306_14011_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu

T, P = I.BC_TRANSMISSIVE, I.BC_PERIODIC
GRIDS = [I.grid2d(5, 3, 1.0, 1.0, T), I.grid2d(304, 128, 1.0, 1.0), I.grid2d(305, 128, 1.0, 1.0, T),
         I.grid2d(256, 256, 1.0, 1.0), I.grid2d(257, 256, 1.0, 1.0, T), I.grid2d(609, 256, 1.0, 1.0),
         I.grid2d(456, 608, 1.0, 1.0, T), I.grid2d(481, 608, 1.0, 1.0),
         I.grid3d(32, 32, 38, 1.0, 1.0, 1.0), I.grid3d(33, 32, 38, 1.0, 1.0, 1.0, T), I.grid3d(64, 38, 32, 1.0, 1.0, 1.0),
         I.grid3d(65, 39, 32, 1.0, 1.0, 1.0, ((P, P), (T, T), (P, P)))]


@pytest.mark.parametrize("g", GRIDS, ids=lambda g: "x".join(map(str, g.n[:g.dim])))
def test_the_chosen_tiles_give_the_default_launchs_bits(g):
    U0 = torch.from_numpy(I.random_smooth(g, seed=3)).cuda()
    out = []
    for launch in (None, fv.fv_default_launch(g)):
        with fv.Solver(g, launch=launch) as s:
            U = U0.clone()
            R = s.residual(U).clone()
            dt0 = s.time_step(U)
            dt = s.rk_step(U, return_dt=True)
            assert dt == dt0  # the step's own reduction and fv_time_step's
            t = s.run(U, 19, return_time=True)
            out.append((R, U, dt, t))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert out[0][2:] == out[1][2:]


@pytest.mark.parametrize("n", [128, 256])
def test_a_nonphysical_cell_is_reported_at_either_reduction(n):
    g, U0 = I.isentropic_vortex(n, seed=0)
    U = torch.from_numpy(U0).cuda()
    U[0, n // 2, n - 1] = -1.0
    with fv.Solver(g) as s:
        with pytest.raises(fv.FvError) as e:
            s.run(U, 1, return_time=True)
        assert e.value.status == fv.FV_ENONPHYSICAL
