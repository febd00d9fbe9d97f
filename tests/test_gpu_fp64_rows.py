"""The FP64 products on both sides of the rule that batches their loads (few warps or
long rows: batched; many short rows: not), with lengths around the batch of 256 entries:
loss and gradient against the FP64 oracle's risk sums and plain matrix products."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p,k", [(300, 255, 1), (300, 256, 2), (257, 1025, 1), (2500, 31, 3), (2499, 600, 4),
                                   (20_000, 33, 1), (20_000, 2, 2), (9, 2501, 2), (3, 30_000, 1)])
def test_loss_and_gradient(n, p, k):
    import paper_2010_16114_gb300 as P
    from paper_2010_16114_gb300.cox import CoxProblem
    P.build()
    rng = np.random.default_rng(n + p)
    X = rng.normal(size=(n, p))
    y, d = rng.exponential(size=n), (rng.random(n) < 0.6).astype(np.uint8)
    d[0] = 1
    B = rng.normal(size=(k, p)) * (0.5 / np.sqrt(p))
    with CoxProblem(X, y, d, precision="fp64") as prob:
        loss, grad = prob.loss_grad(torch.tensor(B, device="cuda"))
        G = grad.cpu().numpy()
        eta = prob.eta(torch.tensor(B, device="cuda")).cpu().numpy()
        _, order = prob.mu_order()
    for c in range(k):
        want = X @ B[c]
        # sums of p (n) products in FP64: 2^-53 times their number, of the sum of magnitudes
        assert np.all(np.abs(eta[c] - want[order]) <= 2.0 ** -52 * (p + 64) * (np.abs(X) @ np.abs(B[c]))[order])
        _, u, f = oracle.risk(y, d, want)
        g = -(d - u) @ X / n
        assert abs(loss[c] - f) <= 1e-12 * max(abs(f), 1.0)
        assert np.linalg.norm(G[c] - g) <= 1e-11 * np.linalg.norm(np.abs(d - u) @ np.abs(X) / n)
