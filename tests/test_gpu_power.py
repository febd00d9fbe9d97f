"""The power method on the genotype tiles (digits of v and X_c v on the
tensor-core products) against numpy in FP64: single tiles, ragged tails, many
partial slots, entries over many magnitudes, and a fixed number of iterations so
that both sides stop at the same estimate."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p", [(1, 1), (17, 9), (1000, 129), (1024, 1024), (3001, 5003), (40_007, 130)])
@pytest.mark.parametrize("start", ["ones", "wide"])
def test_power_method_fixed_iterations(n, p, start):
    from paper_2010_16114_gb300 import _lib as L
    from paper_2010_16114_gb300.cox import CoxProblem
    rng = np.random.default_rng(n + p)
    X = rng.binomial(2, rng.uniform(0.05, 0.5, p), size=(n, p)).astype(np.uint8)
    Xc = X - X.mean(axis=0)
    v = np.ones(p) if start == "ones" else rng.normal(size=p) * 10.0 ** rng.uniform(-6, 0, size=p)
    iters = 4
    u, s = v / np.linalg.norm(v), 0.0
    for _ in range(iters):
        b = Xc.T @ (Xc @ u)
        s = np.linalg.norm(b)
        if s == 0:
            break
        u = b / s
    y = np.arange(n, dtype=np.float64)
    d = np.zeros(n, np.uint8)
    d[::3] = 1
    with CoxProblem(X, y, d) as prob:
        got = prob.lipschitz(None if start == "ones" else v, tol=1e-15, maxiter=iters)
        vp = None if start == "ones" else v.ctypes.data_as(ctypes.c_void_p)
        rc, again = L.cox_lipschitz_noalloc(prob.h, vp, 1e-15, iters)
        assert rc == L.COX_OK and again == got
    # v, X_c v and X_c^T X_c v are rounded to FP32 (2^-24) once each per iteration
    assert abs(got - 2.0 * s / n) <= 2e-6 * max(2.0 * s / n, 1e-6)
