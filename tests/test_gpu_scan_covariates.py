"""The fused scans with unpenalised covariates, at the edges of their variants: 1, 2, 4
and 8 subjects per lane (n up to 64,000, 128,000, 256,000, beyond) and 1..4, 5..8, 9..16
covariates (each count's sums leave from other lanes, and 9..12 skip the last four),
loss and both gradients against the FP64 oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["split_e4m3", "split_e2m1", "fp64", "fp32_gemv"])
@pytest.mark.parametrize("q", [1, 3, 4, 5, 8, 9, 12, 13, 16])
@pytest.mark.parametrize("n", [33, 64_001, 131_073, 256_001])
def test_loss_and_gradients(n, q, precision):
    import paper_2010_16114_gb300 as P
    from paper_2010_16114_gb300.cox import CoxProblem
    P.build()
    rng = np.random.default_rng(100 * q + n % 97)
    k, p = 2, 5
    X = rng.binomial(2, 0.3, size=(n, p)).astype(np.uint8)
    Xf = X.astype(np.float64)
    y, d = np.ceil(rng.uniform(0, 900, n)), (rng.random(n) < 0.3).astype(np.uint8)
    Z = rng.normal(size=(n, q)) * 0.5
    Z[:, 0] = Z[:, 0] > 0
    B, G = rng.normal(size=(k, p)) * 0.2, rng.normal(size=(k, q)) * 0.3
    with CoxProblem(Xf if precision == "fp64" else X, y, d, precision=precision, center=True) as prob:
        b = torch.tensor(B, dtype=prob.dtype, device="cuda")
        B = b.cpu().numpy().astype(np.float64)
        prob.set_covariates(Z)
        prob.set_gamma(G, k)
        loss, grad = prob.loss_grad(b)
        gg = prob.grad_gamma(k)
        grad = grad.cpu().numpy().astype(np.float64)
    mu = Xf.mean(axis=0)
    for c in range(k):
        _, u, f = oracle.risk(y, d, Xf @ B[c] - mu @ B[c] + Z @ G[c])
        v = d - u
        g, gz = -(v @ Xf - v.sum() * mu) / n, -(v @ Z) / n
        # the other covariate tests' gates, of the largest the data could give
        assert abs(loss[c] - f) <= 1e-7 * max(abs(f), 1e-3 * d.mean()), (c, loss[c], f)
        assert np.linalg.norm(grad[c] - g) <= 1e-5 * (np.linalg.norm(g) + np.sqrt(d.sum()) / n), (c, grad[c], g)
        assert np.linalg.norm(gg[c] - gz) <= 1e-5 * (np.linalg.norm(gz) + np.sqrt(d.sum()) / n), (c, gg[c], gz)
