"""What a row's score depends on: its own features, and which side of 8192 rows the
call is on (in integers from there on, an FP64 chain below), nothing else.  On one
side the bits are the same in any call; across it two evaluations differ by at
most the bounds of both (test_gpu_mlp_predict.py)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from test_gpu_mlp_predict import exact, network, predict  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[14, 128, 64, 32, 1], [9, 63, 65, 47, 1]])
def test_scores_across_the_8192_row_line(sizes):
    rng = np.random.default_rng(8)
    layers, X = network(rng, sizes), rng.normal(size=(20000, sizes[0]))
    few, many = predict(sizes, layers, X[:8191]), predict(sizes, layers, X[:8192])
    assert np.array_equal(few[5:300], predict(sizes, layers, X[5:300]))
    assert np.array_equal(many, predict(sizes, layers, X)[:8192])
    assert np.array_equal(many[3:], predict(sizes, layers, X[3:19000])[:8189])
    _, tol = exact(sizes, layers, X[:200])
    assert np.all(abs(few[:200] - many[:200]) <= 2 * tol)
