"""Cells that are all physical, but so rough that the reconstruction leaves face
states of negative pressure.  The flux of such a face is what the method's own
formulas give: a number, or NaN where c~^2 is negative.  Residuals against the
oracle, NaN included, through the fused, marching, split and batched kernels and
the no-alloc entry.

Tolerance, per cell and variable: a flux near c~^2 = 0 is ill-conditioned, so the
scale is what the residual (in extended precision) moves by when the states are
perturbed by 2^-50, the largest of four such changes times 16, beside 8 ulps of
the cell's terms and 1e-12 of the largest residual.  Cells whose NaN comes or
goes under the perturbations are left out."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_2306_14011_gb300 import fv  # noqa: E402
from paper_2306_14011_gb300 import inputs as I  # noqa: E402
from test_gpu_parity import EPS, TOL_RES, dev  # noqa: E402

pytestmark = pytest.mark.gpu


def rough(g, seed):
    rng = np.random.default_rng(seed)
    u = lambda a, b: rng.uniform(a, b, g.shape[1:])  # noqa: E731
    return I.conserved(u(0.2, 4.5), tuple(u(-3, 3) for _ in range(g.dim)), u(0.2, 4.5))


class Expected:
    def __init__(self, g, U, s):
        rng = np.random.default_rng(1)
        self.R = O.residual_ext(g, U, s)
        self.clear = np.ones(U.shape, bool)
        moved = np.zeros(U.shape)
        with np.errstate(invalid="ignore"):
            for _ in range(4):
                P = O.residual_ext(g, U * (1 + 2.0 ** -50 * rng.uniform(-1, 1, U.shape)), s)
                self.clear &= np.isnan(P) == np.isnan(self.R)
                moved = np.fmax(moved, abs(P - self.R))
            terms = np.nan_to_num(O.residual_terms(g, U, s), nan=0.0)
            self.tol = 16 * moved + 8 * EPS * terms + TOL_RES * np.nanmax(abs(self.R))

    def check(self, R):
        assert self.clear.mean() > 0.999
        assert np.array_equal(np.isnan(R)[self.clear], np.isnan(self.R)[self.clear])
        ok = self.clear & ~np.isnan(self.R)
        assert np.all(abs(R - self.R)[ok] <= self.tol[ok])


@pytest.mark.parametrize("lim", [fv.FV_LIM_MINMOD, fv.FV_LIM_VANLEER, fv.FV_LIM_NONE])
@pytest.mark.parametrize("recon", [fv.FV_RECON_CONSERVED, fv.FV_RECON_PRIMITIVE])
@pytest.mark.parametrize("dim", [2, 3])
def test_the_residual_equals_the_oracles_nan_included(dim, recon, lim):
    T = I.BC_TRANSMISSIVE
    g = I.grid2d(397, 401, 1.0, 1.0, T) if dim == 2 else I.grid3d(61, 47, 53, 1.0, 1.0, 1.0)
    U = rough(g, 10 * dim + lim)
    want = Expected(g, U, O.scheme(limiter=lim, recon=recon))
    if recon == fv.FV_RECON_CONSERVED:
        assert np.isnan(want.R).any()  # such faces are there
    for mode in (fv.FV_FUSED, fv.FV_SPLIT):
        with fv.Solver(g, limiter=lim, recon=recon, mode=mode) as s:
            R = s.residual(dev(U))
            want.check(R.cpu().numpy())
            if mode == fv.FV_FUSED:
                N = torch.empty_like(R)
                fv.fv_residual_noalloc(g, s.scheme, dev(U), N)
                torch.cuda.synchronize()
                assert np.array_equal(N.cpu().numpy(), R.cpu().numpy(), equal_nan=True)


def test_the_marching_kernel_too():
    g = I.grid3d(64, 45, 48, 1.0, 1.0, 1.0)
    U = rough(g, 5)
    want = Expected(g, U, O.scheme())
    d = fv.launch_to_dict(fv.fv_default_launch(g))
    for st in range(3):
        d["stage"][st].update(tile=(16, 15, 8), threads=256, march=1)
    with fv.Solver(g, launch=d) as s:
        want.check(s.residual(dev(U)).cpu().numpy())


def test_a_batch_takes_the_single_grids_steps():
    grids = [I.grid2d(97, 130, 1.0, 1.0, I.BC_TRANSMISSIVE), I.grid2d(75, 61, 1.0, 1.0)]
    Us = [rough(g, 3 + i) for i, g in enumerate(grids)]
    with fv.Solver(grids) as s:
        P = s.pack([dev(U) for U in Us])
        s.run(P, 1, 1e-4)
        got = [x.cpu().numpy() for x in s.unpack(P)]
    for g, U, G in zip(grids, Us, got):
        with fv.Solver(g) as s:
            V = dev(U)
            s.rk_step(V, 1e-4)
        assert np.isnan(G).any() and np.array_equal(G, V.cpu().numpy(), equal_nan=True)
