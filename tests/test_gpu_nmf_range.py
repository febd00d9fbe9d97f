"""NMF factors and products near the ends of FP32's range: the APG step 1 / (2 ||G||_F^2
+ eps) where the squares pass FP32's largest or smallest value (they are summed in pairs
of floats), and products that overflow, which are reported."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _nmf(X, r):
    import paper_2010_16114_gb300 as P
    from paper_2010_16114_gb300.nmf import NMF
    P.build()
    return NMF(X, r)


@pytest.mark.parametrize("vs,ws", [(1.0, 1.0), (1e-9, 1e9), (1e9, 1e-9), (1e-12, 1e-12), (3e7, 3e7)])
@pytest.mark.parametrize("algo", ["apg", "mult"])
def test_scaled_factors(algo, vs, ws):
    """V and W scaled by powers so that ||G||_F^2 spans 1e-40 .. 1e43."""
    m, n, r = 300, 500, 7
    X, V0, W0 = synth.nmf_inputs(m, n, r)
    V0, W0 = (V0 * np.float32(vs)).astype(np.float32), (W0 * np.float32(ws)).astype(np.float32)
    Ve, We = oracle.nmf(X, V0, W0, 1, algo, 1e-10)
    if not (np.abs(Ve).max() < 1e30 and np.abs(We).max() < 1e30):
        pytest.skip("the iterate itself leaves FP32")
    h = _nmf(X, r)
    h.set_factors(V0, W0)
    h.iterate(1, algo)
    V, W = h.factors()
    h.close()
    # as the elementwise test of one iteration, with the operands' own size as the floor: the
    # APG step subtracts nearly equal terms of the size of the factor it starts from
    for got, want, start in ((V, Ve, V0), (W, We, W0)):
        floor = np.abs(start).max() if algo == "apg" else 0.0
        assert np.all(np.abs(got - want) <= 2e-5 * np.maximum(np.abs(want), floor)), np.abs(got - want).max()


@pytest.mark.parametrize("algo", ["apg", "mult"])
@pytest.mark.parametrize("m,n", [(130, 20_000), (20_000, 130), (700, 700)])
def test_overflowing_product_is_reported(algo, m, n):
    """X W^T (or X^T V) past FP32's largest value: row tiles of one slot and of many."""
    from paper_2010_16114_gb300 import _lib as L
    X = np.full((m, n), 2.0 ** 124, np.float32)
    h = _nmf(X, 4)
    h.set_factors(np.ones((m, 4), np.float32), np.ones((4, n), np.float32))
    h.iterate(1, algo)
    with pytest.raises(L.CoxError) as e:
        h.sync()
    assert e.value.code == L.COX_ERR_NONFINITE
    h.close()


@pytest.mark.parametrize("r", [3, 20, 80])
def test_gram_sums_past_fp32(r):
    """Gram partials that are finite in FP32 while their sum is not: the sum is finite in
    FP64, and the update takes the FP32 infinity of it (V -> 0 for finite products)."""
    m, n = 200, 12_800
    X = np.full((m, n), 1.0, np.float32)
    h = _nmf(X, r)
    W0 = np.full((r, n), np.float32(1.5e18))  # 32 columns: 7.2e37 a partial, 400 blocks: 2.9e40
    h.set_factors(np.ones((m, r), np.float32), W0)
    f = h.objective()
    # ||X - V W||^2 with every entry (1.5e18 r)^2 to rounding
    want = float(m) * n * (1.5e18 * r) ** 2
    assert any(abs(f - s * want) <= 1e-5 * s * want for s in (0.5, 1.0)), (f, want)
    h.close()


def test_objective_between_iterations():
    """The objective after every mix of iterations, set_factors and repeated calls is that
    of the factors now held (W's Gram matrix is formed late)."""
    m, n, r = 400, 900, 9
    X, V0, W0 = synth.nmf_inputs(m, n, r)
    h = _nmf(X, r)

    def check():
        V, W = h.factors()
        want = oracle.nmf_objective(X, V, W)
        for _ in range(2):
            assert abs(h.objective() - want) <= 1e-5 * want

    h.set_factors(V0, W0)
    check()
    for algo, iters in (("mult", 1), ("apg", 2), ("mult", 0), ("mult", 3)):
        h.iterate(iters, algo)
        check()
    h.set_factors(V0 * 0.5, W0)
    check()
    h.iterate(1, "apg")
    h.set_factors(V0, W0 * 2)
    check()
    h.close()
