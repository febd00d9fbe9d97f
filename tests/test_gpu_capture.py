"""Iterations captured in a CUDA graph: the caller's penalties are read at every replay
(the copy is a node of the graph), in every arithmetic and for more columns than a
kernel argument holds, and the Python front end keeps the array that a replay reads."""
import ctypes
import gc

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N, P = 700, 300


def _data():
    rng = np.random.default_rng(0)
    X = rng.binomial(2, 0.3, (N, P)).astype(np.uint8)
    return X, rng.exponential(size=N), (rng.random(N) < 0.5).astype(np.uint8)


def _problem(precision):
    import paper_2010_16114_gb300 as pkg
    from paper_2010_16114_gb300.cox import CoxProblem
    pkg.build()
    X, y, d = _data()
    return CoxProblem(X.astype(np.float64) if precision == "fp64" else X, y, d, precision=precision, center=True)


CASES = [("split_e4m3", 2), ("split_e2m1", 2), ("fp64", 2), ("fp32_gemv", 2), ("split_e4m3", 20), ("fp64", 70)]


@pytest.mark.parametrize("from_eta", [False, True])
@pytest.mark.parametrize("precision,k", CASES)
def test_replay_reads_the_penalties_anew(precision, k, from_eta):
    from paper_2010_16114_gb300 import _lib as L
    if from_eta and precision == "fp32_gemv":
        pytest.skip("no step from a given eta in the FP32 baseline")
    lib = L.load()
    with _problem(precision) as prob:
        b0 = torch.zeros((k, P), dtype=prob.dtype, device="cuda")
        b0[:, ::7] = 0.05
        eta = None if precision == "fp32_gemv" else prob.eta(b0)
        lam = np.full(k, 0.001)

        def call(b, stream):
            vp = ctypes.c_void_p
            lp = lam.ctypes.data_as(vp)
            if from_eta:
                return lib.cox_prox_step_eta(prob.h, vp(b.data_ptr()), vp(eta.data_ptr()), lp, k, ctypes.c_double(0.5),
                                             vp(stream))
            return lib.cox_prox_step(prob.h, vp(b.data_ptr()), lp, k, ctypes.c_double(0.5), vp(stream))

        want = []
        for v in (0.001, 0.02, 0.0):
            lam[:] = v
            b = b0.clone()
            assert call(b, torch.cuda.current_stream().cuda_stream) == 0
            torch.cuda.synchronize()
            want.append(b)
        lam[:] = 0.001
        b = b0.clone()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            assert call(b, torch.cuda.current_stream().cuda_stream) == 0
        for v, w in zip((0.001, 0.02, 0.0), want):
            lam[:] = v
            b.copy_(b0)
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(b, w), v
        prob.sync()


@pytest.mark.parametrize("explicit", [False, True])
def test_front_end_keeps_what_a_replay_reads(explicit):
    with _problem("split_e4m3") as prob:
        b0 = torch.zeros((3, P), device="cuda")
        b0[:, ::7] = 0.05
        want = []
        for v in (0.004, 0.02):
            b = b0.clone()
            prob.prox_step(b, [v] * 3, 0.5)
            want.append(b)
        torch.cuda.synchronize()
        own = np.full(3, 0.004)
        graphs = []
        for lam in ([0.004] * 3, own):
            b = b0.clone()
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                prob.prox_step(b, lam, 0.5, stream=torch.cuda.current_stream() if explicit else None)
            graphs.append((g, b))
        gc.collect()
        junk = [np.full(3, 1e6) for _ in range(1000)]  # reuses a freed array's memory
        own[:] = 0.02  # the caller's own array: replays follow it
        for (g, b), w in zip(graphs, want):
            b.copy_(b0)
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(b, w)
        del junk
