"""The surrogate's forward pass on the integer pipes (and, for wide networks, in
FP64) over ragged row counts and widths, and on data whose sums leave the
integer path: features and weights far apart in scale, zeros, subnormal
numbers, infinities and NaN.

Tolerance: an FP64 chain of K products and a bias differs from the exact sum by
at most (K + 2) 2^-52 sum |x w| + |b| of it, twice the unit roundoff; an
activation's error d adds |w| d to the next layer's sums."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2306_14011_gb300 import fv  # noqa: E402

pytestmark = pytest.mark.gpu


def exact(sizes, layers, X):
    """The outputs in extended precision and the error bound of an FP64 pass."""
    a, d = X.astype(np.longdouble), np.zeros(X.shape, np.longdouble)
    for l, (W, b) in enumerate(layers):
        W, b = W.astype(np.longdouble), b.astype(np.longdouble)
        d = d @ abs(W) + (len(W) + 2) * 2.0 ** -52 * ((abs(a) + d) @ abs(W) + abs(b))
        a = a @ W + b
        if l < len(layers) - 1:
            a = np.maximum(a, 0)
    return a[:, 0], d[:, 0]


def predict(sizes, layers, X):
    P = torch.from_numpy(np.concatenate([p.ravel() for Wb in layers for p in Wb])).cuda()
    out = torch.full((len(X),), -7.0, dtype=torch.float64, device="cuda")
    fv.fv_mlp_predict(sizes, P, torch.from_numpy(X).cuda(), out)
    return out.cpu().numpy()


def network(rng, sizes):
    return [(rng.normal(size=(i, o)) / np.sqrt(i), rng.normal(size=o)) for i, o in zip(sizes[:-1], sizes[1:])]


# the first four in integers from 8192 rows on
@pytest.mark.parametrize("sizes", [[14, 128, 64, 32, 1], [9, 63, 65, 47, 1], [1, 47, 113, 1], [30, 77, 77, 2, 31, 129, 1],
                                   [1, 1], [1024, 1], [5, 16, 256, 257, 1]])
@pytest.mark.parametrize("n", [1, 8191, 8192, 8209])
def test_outputs_are_within_an_fp64_pass_of_the_exact_ones(sizes, n):
    rng = np.random.default_rng(n)
    layers, X = network(rng, sizes), rng.normal(size=(n, sizes[0]))
    X[0] = 0.0
    got, some = predict(sizes, layers, X), np.unique(np.r_[0:min(n, 20), max(0, n - 40):n, rng.integers(0, n, 100)])
    ref, tol = exact(sizes, layers, X[some])
    assert np.all(abs(got[some] - ref) <= tol)


@pytest.mark.parametrize("spread", [8, 20, 30, 60, 400])
def test_scales_far_apart(spread):
    """Features of scale 2^+-spread that meet weights of the inverse scale."""
    rng = np.random.default_rng(spread)
    sizes = [14, 128, 64, 32, 1]
    layers, X = network(rng, sizes), rng.normal(size=(8200, 14))
    scale = 2.0 ** rng.integers(-spread, spread + 1, size=14)
    X *= scale
    layers[0] = (layers[0][0] / scale[:, None], layers[0][1])
    X[::7, :7] = 0.0
    X[3] *= 2.0 ** -1000
    got, (ref, tol) = predict(sizes, layers, X)[:200], exact(sizes, layers, X[:200])
    assert np.all(abs(got - ref) <= tol + 2.0 ** -1000)


def test_infinities_and_nan_reach_the_rows_they_are_in():
    rng = np.random.default_rng(5)
    sizes = [14, 128, 64, 32, 1]
    layers, X = network(rng, sizes), rng.normal(size=(8192, 14))
    clean = predict(sizes, layers, X)
    X[3, 2], X[20, 0] = np.nan, np.inf
    got = predict(sizes, layers, X)
    rest = np.delete(np.arange(8192), [3, 20])
    assert np.isnan(got[3]) and not np.isfinite(got[20])
    assert np.array_equal(got[rest], clean[rest])
