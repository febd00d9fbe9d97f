"""The fused risk-set scans at the edges of their chunks and tiles: subjects per
lane 1, 2, 4, 8 (n up to 64,000, 128,000, 256,000, beyond), ragged tails, event
groups that fill, miss or cross tiles of 256 (distinct times, whole days, one
group, one event at either end), many tied events, and linear predictors whose
risk-set reciprocals leave FP32's range, against the FP64 oracle."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _times(kind, n, rng):
    if kind == "distinct":
        return rng.permutation(n).astype(np.float64), (rng.random(n) < 0.6).astype(np.uint8)
    if kind == "days":
        return np.ceil(rng.uniform(0, 700, n)), (rng.random(n) < 0.2).astype(np.uint8)
    if kind == "one_time":
        return np.full(n, 3.0), (rng.random(n) < 0.5).astype(np.uint8)
    d = np.zeros(n, np.uint8)
    d[0 if kind == "first" else -1] = 1  # one event, at the earliest or the latest time
    return np.arange(n, dtype=np.float64), d


def _check(n, kind, scale, precision, k=2, p=5):
    from paper_2010_16114_gb300.cox import CoxProblem
    rng = np.random.default_rng(n + len(kind))
    X = rng.binomial(2, 0.3, size=(n, p)).astype(np.uint8)
    y, d = _times(kind, n, rng)
    Xf = X.astype(np.float64)
    B = (rng.normal(size=(k, p)) * scale).astype(np.float32)
    Xin, dt = (Xf, torch.float64) if precision == "fp64" else (X, torch.float32)
    with CoxProblem(Xin, y, d, precision=precision, center=True) as prob:
        loss, grad = prob.loss_grad(torch.tensor(B, dtype=dt, device="cuda"))
        G = grad.cpu().numpy().astype(np.float64)
    mu = Xf.mean(axis=0)
    for c in range(k):
        eta = oracle.eta(Xf, mu, B[c].astype(np.float64))
        _, u, f = oracle.risk(y, d, eta)
        g = -oracle.grad(Xf, mu, d, u)
        # loss within 1e-7, gradient within 1e-5 of the largest the data could give
        # (a single event's gradient may cancel to nearly zero)
        top = np.linalg.norm(g) + np.sqrt(d.sum()) / n
        assert abs(loss[c] - f) <= 1e-7 * max(abs(f), 1e-3 * d.mean()), (c, loss[c], f)
        assert np.linalg.norm(G[c] - g) <= 1e-5 * top, (c, G[c], g)


@pytest.mark.parametrize("kind", ["distinct", "days", "one_time"])
@pytest.mark.parametrize("n", [1, 31, 33, 257, 4096, 64_000, 64_001, 131_073, 256_001])
def test_chunks_and_tiles(n, kind):
    _check(n, kind, 0.3, "split_e2m1" if n % 2 else "split_e4m3")


# a single event at either end leaves V of one entry near 1 and the rest near 1/n
# (or all near 0), below the operand forms' quantum: FP64 handles only
@pytest.mark.parametrize("precision,kind", [("fp64", "days"), ("fp64", "first"), ("fp64", "last"), ("fp32_gemv", "days")])
@pytest.mark.parametrize("n", [33, 4096, 70_001])
def test_other_modes(n, precision, kind):
    _check(n, kind, 0.3, precision)


def test_reciprocals_beyond_fp32():
    """eta falls by about 100 along the time order, so the late risk sets sum to
    ~1e-43 and F passes FP32's largest value while every u stays of order one."""
    from paper_2010_16114_gb300.cox import CoxProblem
    n, p = 2000, 50
    X = np.zeros((n, p), np.uint8)
    for j in range(p):
        X[: n - j * (n // p), j] = 2
    y = np.arange(n, dtype=np.float64)
    d = np.ones(n, np.uint8)
    B = np.full((1, p), 0.98, np.float32)
    Xf = X.astype(np.float64)
    mu = Xf.mean(axis=0)
    with CoxProblem(X, y, d) as prob:
        loss, grad = prob.loss_grad(torch.tensor(B, device="cuda"))
    eta = oracle.eta(Xf, mu, B[0].astype(np.float64))
    _, u, f = oracle.risk(y, d, eta)
    g = -oracle.grad(Xf, mu, d, u)
    # w = exp(eta - max) in FP32: below 2^-126 its spacing is 2^-149, so the smallest
    # w (about e^-98) carries ~2% and its weight in the loss is 1/n per subject
    assert np.isfinite(loss[0]) and abs(loss[0] - f) <= 1e-3 * abs(f)
    assert np.linalg.norm(grad.cpu().numpy()[0] - g) <= 5e-2 * np.linalg.norm(g)
