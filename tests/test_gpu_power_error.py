"""Accuracy of the power method on the genotype tiles against numpy in FP64: what is left
is the FP32 rounding of the products' partial sums, whose errors average out over the
entries (2^-25 of sums a few times the centred ones, over the square root of p = 1,000 or
n = 30,000: 5e-10); v, X_c v and their norms are held to 2^-30 of the largest entry."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_rms_error_of_the_estimate():
    import paper_2010_16114_gb300 as P
    from paper_2010_16114_gb300.cox import CoxProblem
    P.build()
    n, p, iters = 30_000, 1_000, 12
    err = []
    for seed in range(8):
        rng = np.random.default_rng(seed)
        X = rng.binomial(2, rng.uniform(0.05, 0.5, p), size=(n, p)).astype(np.uint8)
        C = X - X.mean(axis=0)
        G = C.T @ C
        v = rng.normal(size=p)
        u = v / np.linalg.norm(v)
        for _ in range(iters):
            b = G @ u
            s = np.linalg.norm(b)
            u = b / s
        y, d = np.arange(n, dtype=np.float64), np.ones(n, np.uint8)
        with CoxProblem(X, y, d) as prob:
            err.append(prob.lipschitz(v, tol=1e-15, maxiter=iters) / (2.0 * s / n) - 1.0)
    # three times the estimate above
    assert np.sqrt(np.mean(np.square(err))) <= 1.5e-9, err
