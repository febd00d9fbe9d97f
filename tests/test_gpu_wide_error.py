"""Rounding of the wide form of the genotype products (ten e2m1 digits per
coefficient) beside the e4m3 kernel's on the same coefficients: both hold the same
values and sum them exactly inside a window, so what differs is how a window's limb
sums are joined, and the wide form's gradients may be no further from FP64.

The long dimension is the second product's, where the uncentred sums are much
larger than the gradient and every rounding counts."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 3, 8])
def test_gradient_error_no_larger_than_the_e4m3_kernels(k):
    import paper_2010_16114_gb300 as P
    from paper_2010_16114_gb300.cox import CoxProblem
    P.build()
    rng = np.random.default_rng(7)
    n, p = 150_001, 401
    X = rng.binomial(2, rng.uniform(0.05, 0.5, p), size=(n, p)).astype(np.uint8)
    Xf = X.astype(np.float64)
    mu = Xf.mean(axis=0)
    y, d = np.ceil(rng.uniform(0, 3000, n)), (rng.random(n) < 0.2).astype(np.uint8)
    kw = (dict(), dict(issue=1))  # the wide form; the e4m3 kernel, as a shape is forced
    sq = np.zeros(2)
    with CoxProblem(X, y, d, **kw[0]) as wide, CoxProblem(X, y, d, **kw[1]) as e4m3:
        for _ in range(8 // k + 1):
            B = (rng.normal(size=(k, p)) * 0.02).astype(np.float32)
            grads = [prob.loss_grad(torch.tensor(B, device="cuda"))[1].cpu().numpy().astype(np.float64)
                     for prob in (wide, e4m3)]
            for c in range(k):
                b = B[c].astype(np.float64)
                _, u, _ = oracle.risk(y, d, Xf @ b - mu @ b)
                v = d - u
                g = -(v @ Xf - v.sum() * mu) / n
                sq += [np.sum((G[c] - g) ** 2) for G in grads]
    # sums of at least 8 x 401 squared roundings: the ratio of two such root mean squares
    # scatters by 1 / sqrt(2 x 3208) = 1.3% where they are independent; three times that
    assert np.sqrt(sq[0]) <= 1.04 * np.sqrt(sq[1]), np.sqrt(sq[0] / sq[1])
