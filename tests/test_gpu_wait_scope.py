"""cox_options.wait_limit_s limits the waits of the tensor-core products only: work
without such a product (FP64 and FP32 handles, whose scans hold grid barriers of their
own; lambda_max's scans; the power method) runs with any limit, also zero."""
import numpy as np
import pytest

from helpers import dense_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32_gemv"])
@pytest.mark.parametrize("covariates", [False, True])
def test_zero_limit_without_products(precision, covariates):
    import paper_2010_16114_gb300 as P
    from paper_2010_16114_gb300.cox import CoxProblem
    P.build()
    w, X, Xf, mu = dense_problem("geno_100k_50k", n=20_000, p=64)
    dt = torch.float64 if precision == "fp64" else torch.float32
    beta = torch.full((2, w.p), 0.01, dtype=dt, device="cuda")
    out = []
    for limit in (2.0, 0.0):
        with CoxProblem(Xf if precision == "fp64" else X, w.y, w.delta, precision=precision, center=True,
                        wait_limit_s=limit) as prob:
            if covariates:
                prob.set_covariates(np.random.default_rng(1).normal(size=(w.n, 2)))
            res = []
            for _ in range(5):
                loss, grad = prob.loss_grad(beta)
                res.append((loss, grad.cpu().numpy()))
            out.append(res + [prob.lambda_max(), prob.lipschitz(maxiter=3)])
    for a, b in zip(out[0][:5], out[1][:5]):
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    assert out[0][5:] == out[1][5:]


def test_zero_limit_power_method_on_genotypes():
    import paper_2010_16114_gb300 as P
    from paper_2010_16114_gb300.cox import CoxProblem
    P.build()
    w, X, _, _ = dense_problem("geno_100k_50k", n=3000, p=700)
    with CoxProblem(X, w.y, w.delta) as a, CoxProblem(X, w.y, w.delta, wait_limit_s=0.0) as b:
        assert a.lipschitz(maxiter=5) == b.lipschitz(maxiter=5)
