"""The time-step reduction's launch setting on the grids that reduce in one pass
(up to 65536 cells): it acts there as elsewhere, and any setting gives the same
bits -- one CTA, more and fewer CTAs than cells need, on both sides of the 128 CTAs
that the one pass takes, ragged grids.  Exact: a maximum has no order."""
import pytest

torch = pytest.importorskip("torch")

from paper_2306_14011_gb300 import fv  # noqa: E402
from paper_2306_14011_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu

GRIDS = [I.grid2d(5, 3, 1.0, 1.0), I.grid2d(131, 77, 1.0, 1.0), I.grid2d(256, 256, 1.0, 1.0), I.grid2d(257, 256, 1.0, 1.0),
         I.grid3d(33, 19, 21, 1.0, 1.0, 1.0)]


@pytest.mark.parametrize("g", GRIDS, ids=lambda g: "x".join(map(str, g.n[:g.dim])))
def test_every_setting_gives_the_same_step(g):
    U0 = torch.from_numpy(I.random_smooth(g, seed=2)).cuda()
    small = U0[0].numel() <= 65536
    out = []
    with fv.Solver(g) as s:
        first = s.launch
        assert first["dt"] == dict(threads=128 if small else 512, grid=0)
        for threads in (128, 32, 512, 1024):
            for grid in (0, 1, 7, 128, 129, 200):
                s.launch = dict(first, dt=dict(threads=threads, grid=grid))
                U = U0.clone()
                out.append((s.run(U, 3, return_time=True), U))
    assert all(t == out[0][0] and torch.equal(U, out[0][1]) for t, U in out[1:])


def test_split_contexts_keep_their_default():
    g = I.grid2d(64, 64, 1.0, 1.0)
    with fv.Solver(g, mode=fv.FV_SPLIT) as s:
        assert s.launch["dt"] == dict(threads=512, grid=0)
