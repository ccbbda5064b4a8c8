"""Training on one minibatch of sixty million rows: the sums over its rows take
seconds, most of them in one CTA (a network of two parameters), and the others
wait for it.

Tolerance: the loss is a sum of n terms in a fixed order of about n / 256 per
thread and a tree; n 2^-53 of a sum of positive terms is 7e-9."""
import pytest

torch = pytest.importorskip("torch")

from paper_2306_14011_gb300 import fv  # noqa: E402

pytestmark = pytest.mark.gpu


def test_a_batch_of_every_row():
    n = 60_000_000
    X = torch.rand(n, 1, dtype=torch.float64, device="cuda")
    y = 2 * X[:, 0] + 1
    order = torch.arange(n, dtype=torch.int32, device="cuda").reshape(1, n)
    params = torch.tensor([0.3, 0.1], dtype=torch.float64, device="cuda")
    h = fv.mlp_hyper(n_iter_no_change=0, batch=n)
    loss = fv.fv_mlp_train([1, 1], params, X, y, order, h)
    want = 0.5 * ((0.3 * X[:, 0] + 0.1 - y) ** 2).mean().item()
    assert len(loss) == 1 and abs(loss[0] - want) <= 7e-9 * want
    # Adam's first step is lr against the sign of the gradient
    assert params.tolist() == pytest.approx([0.3 + h.lr, 0.1 + h.lr], abs=1e-8)
