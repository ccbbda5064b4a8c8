"""Solver(mode=FV_FUSED) is Solver(): the same launch, single grids and batches."""
import pytest

torch = pytest.importorskip("torch")

from paper_2306_14011_gb300 import fv  # noqa: E402
from paper_2306_14011_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [I.grid2d(128, 128, 1.0, 1.0), I.grid3d(32, 32, 32, 1.0, 1.0, 1.0),
                                  [I.grid2d(70, 90, 1.0, 1.0), I.grid2d(64, 64, 1.0, 1.0)]], ids=["2d", "3d", "batch"])
def test_the_fused_mode_is_the_default(grid):
    with fv.Solver(grid) as a, fv.Solver(grid, mode=fv.FV_FUSED) as b:
        assert a.launch == b.launch


def test_a_given_launch_keeps_its_settings():
    g = I.grid2d(128, 128, 1.0, 1.0)
    want = fv.launch_to_dict(fv.fv_default_launch(g))
    with fv.Solver(g, launch=fv.fv_default_launch(g), mode=fv.FV_FUSED) as s:
        assert s.launch == want
    with fv.Solver(g, mode=fv.FV_SPLIT) as s:
        assert s.launch == dict(want, mode=fv.FV_SPLIT)
