"""A kernel whose shared memory depends on the problem (the adjoint's), launched
from two threads on problems of different needs: a small problem's launch must
not lower the limit that a large one's needs.  Results are compared with a
first pass that ran alone: the same kernels on the same inputs, bit for bit."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2306_14011_gb300 import fv  # noqa: E402
from paper_2306_14011_gb300 import inputs as I  # noqa: E402

pytestmark = pytest.mark.gpu


def adjoint(g):
    U = torch.from_numpy(I.random_smooth(g, seed=1)).cuda()
    lam = torch.randn(U.shape, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(2))

    def go(stream):
        with fv.Solver(g, stream=stream) as s:
            out = torch.empty_like(U)
            s.residual_vjp(U, lam, out)
            fv.fv_sync(s.ctx)
        return out.cpu().numpy()
    return go


def test_launches_of_different_needs_do_not_disturb_each_other():
    work = [adjoint(I.grid2d(24, 24, 1.0, 1.0)), adjoint(I.grid2d(700, 500, 1.0, 1.0))]
    torch.cuda.synchronize()
    alone = [w(torch.cuda.Stream()) for w in work]
    wrong = []

    def run(w, ref):
        stream = torch.cuda.Stream()
        try:
            for _ in range(20):
                if not np.array_equal(w(stream), ref):
                    wrong.append("differs")
        except Exception as e:  # reported by the main thread
            wrong.append(repr(e))

    threads = [threading.Thread(target=run, args=(w, r)) for w, r in zip(work, alone)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong, wrong[:3]
