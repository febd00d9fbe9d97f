"""The objective history behind the stopping rule of a path fit, |F_t - F_(t-lag)| /
|F_t + 1| < tol, in every arithmetic: one entry per iteration, each the F that a
step-by-step run reports, also when the last run of iterations is shorter than the lag
(the ring of the runs before must then still hold each iteration's own F)."""
import numpy as np
import pytest

from helpers import dense_problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _history(blob, p, k, itemsize):
    o = 64 + k * p * itemsize + 8 * k
    n = int(np.frombuffer(blob, np.int64, 8)[7])
    F = np.frombuffer(blob, np.float64, n, o)
    out = []
    while len(F):
        m = int(F[0])
        out.append(F[1:1 + m])
        F = F[1 + m:]
    return out


@pytest.mark.parametrize("precision", ["fp32_gemv", "split_e4m3", "split_e2m1", "fp64"])
@pytest.mark.parametrize("lag,iters", [(10, 10), (10, 11), (10, 12), (1, 3), (2, 5)])
def test_every_iteration_keeps_its_own_objective(precision, lag, iters):
    import paper_2010_16114_gb300 as P
    from paper_2010_16114_gb300.cox import CoxProblem
    P.build()
    w, X, Xf, mu = dense_problem("geno_100k_50k", n=900, p=300)
    dt = torch.float64 if precision == "fp64" else torch.float32
    lams, step = [0.004, 0.001], 0.4
    with CoxProblem(Xf if precision == "fp64" else X, w.y, w.delta, precision=precision, center=True, lag=lag) as prob:
        b = torch.zeros((2, w.p), dtype=dt, device="cuda")
        want = []
        for _ in range(iters):
            prob.prox_step(b, lams, step)
            want.append(prob.last_objective(2))
        want = np.array(want).T
        fit, it, obj, _ = prob.path_fit(lams, step, max_iter=iters, tol=0.0)
        got = _history(prob.get_state(), w.p, 2, 8 if precision == "fp64" else 4)
        assert list(it) == [iters, iters] and torch.equal(fit, b)
        for c in range(2):
            assert np.array_equal(got[c], want[c]), (c, got[c], want[c])
            assert obj[c] == want[c][-1]


@pytest.mark.parametrize("k,lag,iters", [(3, 700, 702), (200, 10, 11), (64, 28, 30)])
def test_more_results_than_the_small_block(k, lag, iters):
    """Results that do not fit beside the error bits (16 KB with the ring of the path
    fit: lag + 3 values per column) come back the same; (64, 28) just fits."""
    import paper_2010_16114_gb300 as P
    from paper_2010_16114_gb300.cox import CoxProblem
    P.build()
    w, X, Xf, mu = dense_problem("geno_100k_50k", n=200, p=60)
    lams, step = np.linspace(0.02, 0.0, k), 0.4
    with CoxProblem(Xf, w.y, w.delta, precision="fp64", center=True, lag=lag) as prob:
        b = torch.zeros((k, w.p), dtype=torch.float64, device="cuda")
        want = []
        for _ in range(iters):
            prob.prox_step(b, lams, step)
            want.append(prob.last_objective(k))
        want = np.array(want).T
        f, l1 = prob.last_loss_l1(k)
        assert np.array_equal(f + lams * l1, want[:, -1])
        fit, it, obj, _ = prob.path_fit(lams, step, max_iter=iters, tol=0.0)
        got = _history(prob.get_state(), w.p, k, 8)
        assert torch.equal(fit, b) and np.array_equal(np.array(got), want)
        assert np.array_equal(obj, want[:, -1])
        loss, _ = prob.loss_grad(torch.zeros_like(b))
        assert np.ptp(loss) == 0.0 and loss[0] > 0


@pytest.mark.parametrize("precision", ["fp32_gemv", "split_e4m3", "split_e2m1", "fp64"])
def test_loss_and_l1_of_every_column(precision):
    import paper_2010_16114_gb300 as P
    from paper_2010_16114_gb300.cox import CoxProblem
    P.build()
    w, X, Xf, mu = dense_problem("geno_100k_50k", n=900, p=300)
    B = np.random.default_rng(5).normal(size=(3, w.p)) * np.array([[0.01], [0.03], [0.002]])
    lams = [0.01, 0.002, 0.0]
    with CoxProblem(Xf if precision == "fp64" else X, w.y, w.delta, precision=precision, center=True) as prob:
        b = torch.tensor(B, dtype=prob.dtype, device="cuda")
        norms = b.double().abs().sum(1).cpu().numpy()
        loss, _ = prob.loss_grad(b)
        prob.prox_step(b, lams, 0.3)
        f, l1 = prob.last_loss_l1(3)
        assert np.array_equal(f, loss)
        assert np.allclose(l1, norms, rtol=1e-12, atol=0)  # sums of 300 terms in FP64 or pairs of floats
        assert np.allclose(prob.last_objective(3), f + np.array(lams) * l1, rtol=1e-14, atol=0)
