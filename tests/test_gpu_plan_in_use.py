"""What a handle launches, as it reports it: the default plan, a forced one, an autotuned
one; and an autotuner's choice given back as options makes a handle that launches the
same kernel."""
import numpy as np
import pytest

from helpers import dense_problem, oracle_loss_grad, rel_l2

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def data():
    import paper_2010_16114_gb300 as P
    P.build()
    return dense_problem("geno_100k_50k", n=3000, p=2100)


@pytest.mark.parametrize("precision,k", [("split_e4m3", k) for k in (1, 3, 6, 8, 12, 16, 32)] + [("split_e2m1", 8)])
def test_choice_as_options_gives_the_same_kernel(data, precision, k):
    from paper_2010_16114_gb300 import cox
    w, X, Xf, mu = data
    rng = np.random.default_rng(k)
    B = torch.tensor((rng.normal(size=(k, w.p)) * (rng.random((k, w.p)) < 0.03) * 0.05).astype(np.float32), device="cuda")
    with cox.CoxProblem(X, w.y, w.delta, precision=precision) as prob:
        default = cox.default_plan(k, precision)
        assert prob.plan(k) == {"x_b": default, "xt_v": default}
        tune = prob.autotune(k, reps=1)
        plan = prob.plan(k)
        loss, grad = prob.loss_grad(B)
        info = prob.info()
        assert (info["tile_m"], info["chunks"], info["stages"]) == tuple(plan["x_b"][f] for f in ("tile_m", "chunks", "stages"))
    for product in ("x_b", "xt_v"):
        opts = {f: tune[product][f] for f in ("tile_m", "chunks", "stages", "issue")}
        with cox.CoxProblem(X, w.y, w.delta, precision=precision, **opts) as again:
            assert again.plan(k)[product] == plan[product]
            loss2, grad2 = again.loss_grad(B)
            for c in (0, k - 1):
                f, g = oracle_loss_grad(Xf, mu, w.y, w.delta, B[c].cpu().numpy().astype(np.float64))
                assert abs(loss2[c] - f) <= 1e-7 * abs(f) and rel_l2(grad2[c].cpu().numpy(), g) <= 1e-5
            if again.plan(k) == plan:  # both products of one kind: the same numbers
                assert np.array_equal(loss, loss2) and torch.equal(grad, grad2)


def test_forced_shapes_and_other_precisions(data):
    from paper_2010_16114_gb300 import _lib as L
    from paper_2010_16114_gb300.cox import CoxProblem, plan_shape
    w, X, Xf, _ = data
    with CoxProblem(X, w.y, w.delta, issue=1) as prob:
        want = {"form": "e4m3", **plan_shape(3, issue=1)}
        assert prob.plan(3) == {"x_b": want, "xt_v": want}
        with pytest.raises(L.CoxError):
            prob.plan(65)
    with CoxProblem(X, w.y, w.delta, precision="fp32_gemv") as prob:
        with pytest.raises(L.CoxError) as e:
            prob.plan(1)
        assert e.value.code == L.COX_ERR_UNSUPPORTED
