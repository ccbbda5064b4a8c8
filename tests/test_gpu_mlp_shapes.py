"""The surrogate's training kernel over the shapes its mapping turns on: widths
below, at and above a CTA's threads, one layer, one sample, batches of one row
and of more rows than CTAs, ragged last batches.

Tolerance: two epochs of Adam in FP64 on both sides, sums in another order.  A
step moves a parameter by lr m / (sqrt(v) + 1e-9), whose relative error is that
of the gradient, a sum of at most 700 products: 700 * 2^-53 < 1e-13 of the
magnitudes summed, at most some hundred times that where they cancel; times the
steps taken (at most 100) and lr = 9e-4 this stays below 1e-11 of a parameter of
size one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import mlp as M  # noqa: E402
from paper_2306_14011_gb300 import fv  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,n,batch", [([3, 1], 7, 3), ([1, 1, 1], 1, 200), ([14, 300, 40, 1], 90, 31),
                                           ([20, 128, 64, 32, 1], 1200, 700), ([5, 16, 256, 257, 1], 50, 50),
                                           ([4, 2, 2, 2, 2, 2, 2, 2, 1], 40, 1)])
def test_training_matches_the_oracle(sizes, n, batch):
    rng = np.random.default_rng(1)
    X = rng.normal(size=(n, sizes[0]))
    y = np.tanh(X[:, 0]) + 0.1 * rng.normal(size=n)
    init = M.glorot_init(sizes, rng.random(M.n_params(sizes)))
    order = np.stack([rng.permutation(n) for _ in range(2)]).astype(np.int32)
    hyper = dict(batch=batch, n_iter_no_change=1000)
    ref = [p.copy() for p in init]
    losses_ref = M.train(ref, X, y, order, hyper)
    P = torch.from_numpy(np.concatenate([p.ravel() for p in init])).cuda()
    losses = fv.fv_mlp_train(sizes, P, torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda(),
                             torch.from_numpy(order).cuda(), fv.mlp_hyper(**hyper))
    np.testing.assert_allclose(losses, losses_ref, rtol=1e-11)
    np.testing.assert_allclose(P.cpu().numpy(), np.concatenate([p.ravel() for p in ref]), rtol=0, atol=1e-11)
