"""The wide form of the genotype products (an e4m3 handle's coefficients as ten
e2m1 digits each, kind::mxf4), which e4m3 handles take for k <= 12 when no
pipeline shape is forced: loss and gradient against the FP64 oracle at every
limb-column class and at both ends of each, on row groups that span several
accumulation windows, and against the e4m3 kernel on the same coefficients."""
import numpy as np
import pytest

from helpers import dense_problem, oracle_loss_grad, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def data():
    import paper_2010_16114_gb300 as P
    P.build()
    return dense_problem("geno_100k_50k", n=9100, p=8700)


def _betas(p, k, seed):
    rng = np.random.default_rng(seed)
    B = np.zeros((k, p))
    for c in range(k):
        idx = rng.choice(p, 60, replace=False)
        # magnitudes over five decades: small coefficients keep their leading bits
        B[c, idx] = rng.normal(size=60) * 10.0 ** rng.uniform(-5, -0.7, size=60)
    return B.astype(np.float32)


# classes of 16, 32, 64 and 128 limb columns: k = 1 | 2, 3 | 4, 6 | 7, 12
@pytest.mark.parametrize("k", [1, 2, 3, 4, 6, 7, 12])
@pytest.mark.parametrize("window", [16, 0])
def test_wide_loss_grad(data, k, window):
    from paper_2010_16114_gb300.cox import CoxProblem
    w, X, Xf, mu = data
    B = torch.tensor(_betas(w.p, k, 100 + k), device="cuda")
    with CoxProblem(X, w.y, w.delta, precision="split_e4m3", window=window) as prob:
        loss, grad = prob.loss_grad(B)
        G = grad.cpu().numpy()
    # the e4m3 kernel (a forced issue mode) on the same coefficients: the operands'
    # values are equal, only FP32 summation orders differ (2^-24 relative per sum)
    with CoxProblem(X, w.y, w.delta, precision="split_e4m3", window=window, issue=1) as prob:
        loss1, grad1 = prob.loss_grad(B)
        G1 = grad1.cpu().numpy()
    for c in range(k):
        f, g = oracle_loss_grad(Xf, mu, w.y, w.delta, B[c].cpu().numpy().astype(np.float64))
        assert abs(loss[c] - f) <= 1e-7 * abs(f), (c, loss[c], f)
        assert rel_l2(G[c], g) <= 1e-5, (c, rel_l2(G[c], g))
        assert rel_l2(G[c], G1[c]) <= 2e-6, (c, rel_l2(G[c], G1[c]))
        assert abs(loss[c] - loss1[c]) <= 1e-8 * abs(f)


def test_wide_reports_non_finite(data):
    """A NaN coefficient (which the maximum that sets the scale skips) is reported."""
    from paper_2010_16114_gb300 import _lib as L
    from paper_2010_16114_gb300.cox import CoxProblem
    w, X, _, _ = data
    B = torch.tensor(_betas(w.p, 2, 5), device="cuda")
    B[1, 17] = float("nan")
    with CoxProblem(X, w.y, w.delta, precision="split_e4m3") as prob:
        with pytest.raises(L.CoxError) as e:
            prob.loss_grad(B)
        assert e.value.code == L.COX_ERR_NONFINITE
