"""The adjoint kernel over its tiles and its FP64 lanes.

Grids on both sides of each change of tile (adjoint() in fv_api.cu), ragged,
with each boundary: the dot-product identity <lam, J d> = <J^T lam, d> with the
oracle's forward-mode J d, at the 1e-12 of the other identity tests (a rounding
error of 2^-53 per term, of which some hundred enter each of the two sums).
A state scaled so far down that its densities leave the range of the integer
arithmetic (2^-300) is evaluated in FP64 lane by lane: scaling a state and its
perturbation by a power of two scales J d exactly, so the same identity holds."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402
from paper_2306_14011_gb300 import fv  # noqa: E402
from paper_2306_14011_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu

T, P = I.BC_TRANSMISSIVE, I.BC_PERIODIC
GRIDS = [I.grid2d(152, 192, 1.0, 1.0), I.grid2d(153, 193, 1.0, 1.0, T), I.grid2d(227, 385, 1.0, 1.0, T),
         I.grid2d(301, 290, 1.0, 1.0, ((P, P), (T, T), (P, P))), I.grid3d(32, 19, 16, 1.0, 1.0, 1.0, T),
         I.grid3d(33, 29, 27, 1.0, 1.0, 1.0), I.grid3d(65, 57, 61, 1.0, 1.0, 1.0, ((P, P), (P, P), (T, T)))]


def _identity(g, U, lam, d, scale=1.0):
    _, Jd = O.residual_jvp(g, U, d)
    with fv.Solver(g) as s:
        JTl = s.residual_vjp(torch.from_numpy(U * scale).cuda(), torch.from_numpy(lam).cuda()).cpu().numpy()
    assert abs(np.sum(lam * Jd) - np.sum(JTl * d)) <= 1e-12 * np.sum(np.abs(lam * Jd))


def _case(g):
    rng = np.random.default_rng(5)
    U = I.random_smooth(g, seed=4)
    lam = rng.normal(size=U.shape)
    return U, lam, rng.normal(size=U.shape) * np.abs(U).reshape(U.shape[0], -1).mean(axis=1).reshape(
        (U.shape[0],) + (1,) * (U.ndim - 1))


@pytest.mark.parametrize("g", GRIDS, ids=lambda g: "x".join(map(str, g.n[:g.dim])))
def test_dot_product_identity_over_the_tiles(g):
    _identity(g, *_case(g))


@pytest.mark.parametrize("g", [I.grid2d(40, 33, 1.0, 1.0, T), I.grid3d(12, 9, 10, 1.0, 1.0, 1.0)], ids=["2d", "3d"])
def test_states_outside_the_integer_range(g):
    # the flux is homogeneous of degree one: J is the same at the scaled state
    U, lam, d = _case(g)
    _identity(g, U, lam, d, scale=2.0 ** -400)
    with fv.Solver(g) as s:  # the flux itself: R scales with the state
        R1 = s.residual(torch.from_numpy(U).cuda()).cpu().numpy()
        R2 = s.residual(torch.from_numpy(U * 2.0 ** -400).cuda()).cpu().numpy() * 2.0 ** 400
    # two evaluations of a sum of fluxes, a few roundings each: 8 ulps of its terms
    tol = 8 * np.finfo(float).eps * O.residual_terms(g, U).reshape(g.nvar, -1).max(axis=1)
    assert np.all(np.abs(R1 - R2).reshape(g.nvar, -1).max(axis=1) <= tol)
