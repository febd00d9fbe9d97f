"""Non-finite coefficients in every operand form, dense and active-set products: the
column they are in is reported and carries NaN through eta (no form computes it as if
the coefficient were zero), and the other columns are what they are without it."""
import numpy as np
import pytest

from helpers import dense_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def data():
    import paper_2010_16114_gb300 as P
    P.build()
    return dense_problem("geno_100k_50k", n=2500, p=1500)


# the wide form (k = 3), the e4m3 kernel (an issue mode is forced), e2m1, FP32
FORMS = [("split_e4m3", {}), ("split_e4m3", {"issue": 1}), ("split_e2m1", {}), ("fp32_gemv", {})]


@pytest.mark.parametrize("value", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("active", [False, True])
@pytest.mark.parametrize("precision,kw", FORMS)
def test_column_is_reported_and_not_computed(data, precision, kw, active, value):
    from paper_2010_16114_gb300 import _lib as L
    from paper_2010_16114_gb300.cox import CoxProblem
    w, X, _, _ = data
    rng = np.random.default_rng(3)
    B = np.zeros((3, w.p), np.float32)
    for c in range(3):
        B[c, rng.choice(w.p, 40, replace=False)] = rng.normal(size=40) * 0.05
    bad = B.copy()
    bad[1, 17] = value
    lam = [0.001, 0.001, 0.001]
    with CoxProblem(X, w.y, w.delta, precision=precision, active_set=active, **kw) as prob:
        good = torch.tensor(B, device="cuda")
        prob.prox_step(good, lam, 0.3)
        prob.sync()
        with pytest.raises(L.CoxError) as e:
            prob.loss_grad(torch.tensor(bad, device="cuda"))
        assert e.value.code == L.COX_ERR_NONFINITE
        b = torch.tensor(bad, device="cuda")
        prob.prox_step(b, lam, 0.3)
        with pytest.raises(L.CoxError):
            prob.sync()
        # S(NaN) = 0: nothing of the column's step is computed from the other coefficients
        assert not torch.any(b[1] != 0)
        for c in (0, 2):
            # the bad column's support may widen the active set: same sums, another FP32 order
            assert torch.allclose(b[c], good[c], rtol=0, atol=1e-6 if active else 0.0)
        if np.isnan(value) and precision != "fp32_gemv":
            eta = prob.eta(torch.tensor(bad, device="cuda")).cpu().numpy()
            assert np.isnan(eta[1]).all() and np.isfinite(eta[[0, 2]]).all()
        # the handle stays usable
        again = torch.tensor(B, device="cuda")
        prob.prox_step(again, lam, 0.3)
        prob.sync()
        assert torch.allclose(again, good, rtol=0, atol=1e-6 if active else 0.0)
