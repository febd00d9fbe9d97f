"""The calls a user of this package makes, at the sizes they make them, for timing and comparison.

Each case is one pass through a public entry point (``CoxProblem``, ``cox_nll``, ``NMF``) on synthetic
data made on the GPU from a seed: genotypes in Hardy-Weinberg proportions, follow-up in whole days with
ties and censoring (arXiv 2010.16114, Sections 5.3 and 6), nonnegative matrices on the grid k / 256
(Section 5.1).  ``exact`` restates each pass in FP64 with plain torch."""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2010_16114_gb300.autograd import cox_nll
from paper_2010_16114_gb300.cox import CoxProblem
from paper_2010_16114_gb300.nmf import NMF


def listed():
    return [
        # one step on a small dense FP64 design: the paper's simulated Cox data (normal_1k_2k)
        dict(name="fp64_step_1k_2k", kind="fp64_step", n=1000, p=2000, k=1, rate=0.7),
        # a small cohort inside a torch program: loss and gradient through autograd, ragged sizes
        dict(name="autograd_4099_1500_k3", kind="autograd", precision="split_e4m3", n=4099, p=1500, k=3, rate=0.2),
        # a short warm-started fit of one penalty on a candidate-SNP panel (geno_200k_10k)
        dict(name="fit_200k_10k_k1", kind="fit", precision="split_e4m3", n=200_000, p=10_000, k=1, rate=0.2, iters=20),
        # one iteration for one penalty in a user's own loop (geno_100k_50k), the default operand form
        dict(name="step_100k_50k_k1", kind="step", precision="split_e4m3", n=100_000, p=50_000, k=1, rate=0.2,
             active=False),
        # one iteration of a 32-penalty batched path (geno_400k_100k_k32)
        dict(name="step_400k_100k_k32", kind="step", precision="split_e4m3", n=400_000, p=100_000, k=32, rate=0.1,
             active=False),
        # one iteration of the 16-penalty biobank path (the rows of geno_400k_500k_k16, fewer SNPs), e2m1 form
        dict(name="step_400k_200k_k16", kind="step", precision="split_e2m1", n=400_000, p=200_000, k=16, rate=0.05,
             active=False),
        # the sparse end of the path with the active set: 8 penalties, few nonzero coefficients, odd sizes
        dict(name="active_200k_99991_k8", kind="step", precision="split_e2m1", n=199_999, p=99_991, k=8, rate=0.05,
             active=True),
        # the Section 6 workflow: covariates without a penalty, one penalty after another
        dict(name="seq_20k_5k_q11", kind="seq", precision="split_e2m1", n=20_011, p=5_003, k=3, q=11, rate=0.05,
             iters=10),
        # the step size every fit needs: the power method of Section 4.4
        dict(name="lipschitz_100k_50k", kind="lipschitz", precision="split_e4m3", n=100_000, p=50_000, iters=20),
        # NMF at the paper's single-GPU size, multiplicative updates
        dict(name="nmf_10k_10k_r20", kind="nmf", m=10_000, n=10_000, r=20, algo="mult", iters=20),
        # the paper's largest rank, projected gradient, a ragged wide matrix
        dict(name="nmf_3001_8009_r60_apg", kind="nmf", m=3_001, n=8_009, r=60, algo="apg", iters=20),
        # a small factorisation, where launches count
        dict(name="nmf_700_1000_r5", kind="nmf", m=700, n=1_000, r=5, algo="mult", iters=20),
    ]


def _between(rng, lo, hi):
    """A whole number between lo and hi, even over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fp64_step", "autograd", "fit", "step", "step", "step", "active", "seq", "lipschitz", "nmf",
                       "nmf", "nmf"])
    rate = rng.choice([0.05, 0.1, 0.2])
    form = rng.choice(["split_e4m3", "split_e2m1"])
    if kind == "fp64_step":
        return dict(kind=kind, n=_between(rng, 500, 4000), p=_between(rng, 500, 4000), k=rng.randint(1, 4), rate=0.7)
    if kind == "autograd":
        return dict(kind=kind, precision=form, n=_between(rng, 1000, 20_000), p=_between(rng, 129, 5000),
                    k=rng.randint(1, 8), rate=rate)
    if kind == "fit":
        return dict(kind=kind, precision=form, n=_between(rng, 20_000, 200_000), p=_between(rng, 2000, 20_000),
                    k=rng.choice([1, 4, 16]), rate=rate, iters=20)
    if kind == "step":
        n = _between(rng, 20_000, 400_000)
        # at most the codes of the largest listed case, and fewer at the widest batch
        k = rng.choice([1, 3, 8, 16] if form == "split_e2m1" else [1, 3, 8, 16, 32])
        most = min(200_000, int((4e10 if k > 16 else 8e10) / n))
        return dict(kind=kind, precision=form, n=n, p=_between(rng, 5000, most), k=k, rate=rate, active=False)
    if kind == "active":
        return dict(kind="step", precision=form, n=_between(rng, 50_000, 200_000), p=_between(rng, 20_000, 100_000),
                    k=rng.choice([4, 8]), rate=rate, active=True)
    if kind == "seq":
        return dict(kind=kind, precision=form, n=_between(rng, 5000, 50_000), p=_between(rng, 1000, 10_000),
                    k=rng.randint(2, 4), q=rng.choice([1, 3, 11]), rate=rate, iters=10)
    if kind == "lipschitz":
        return dict(kind=kind, precision=form, n=_between(rng, 10_000, 100_000), p=_between(rng, 2000, 50_000), iters=20)
    return dict(kind=kind, m=_between(rng, 300, 10_000), n=_between(rng, 300, 10_000), r=_between(rng, 4, 60),
                algo=rng.choice(["mult", "apg"]), iters=20)


# ---- inputs ---------------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _genotypes(g, n, p):
    """Row-major 2-bit codes (n, ceil(p/4)) on the device: x_ij in {0, 1, 2} with frequencies (1-f)^2,
    2f(1-f), f^2 (to 1/256), f ~ U(.05, .5) per SNP."""
    pb = (p + 3) // 4
    f = torch.empty(4 * pb, device="cuda").uniform_(0.05, 0.5, generator=g)
    f[p:] = 0.0  # codes past p stay 0
    one = torch.round(256 * (1 - (1 - f) ** 2)).to(torch.int16)
    two = torch.round(256 * f * f).to(torch.int16)
    out = torch.empty((n, pb), dtype=torch.uint8, device="cuda")
    rows = max(1, (1 << 28) // (4 * pb))
    for i in range(0, n, rows):
        m = min(rows, n - i)
        u = torch.randint(-2**31, 2**31, (m, pb), dtype=torch.int32, device="cuda", generator=g)
        u = u.view(torch.uint8).view(m, 4 * pb)
        c = (u < one).to(torch.uint8)
        c += u < two
        c = c.view(m, pb, 4)
        out[i:i + m] = c[..., 0] | (c[..., 1] << 2) | (c[..., 2] << 4) | (c[..., 3] << 6)
    return out


def _codes(packed, p, dtype=torch.float64):
    """Codes (rows, p) of packed rows."""
    sh = torch.tensor([0, 2, 4, 6], dtype=torch.uint8, device="cuda")
    c = (packed[..., None] >> sh) & 3
    return c.view(packed.shape[0], -1)[:, :p].to(dtype)


def _survival(g, n, eta, rate, ties):
    """Times and events: T ~ Exp(rate exp(eta)), C ~ U(0, 3650) days, the earlier one seen (in whole days
    with ties), about `rate` of the subjects with an event."""
    d = 3650.0
    if rate >= 0.5:
        mean = d * (1 - rate)
    else:
        mean = d / (2 * rate)
    t = torch.empty(n, dtype=torch.float64, device="cuda").exponential_(1.0, generator=g) * mean * torch.exp(-eta)
    c = torch.empty(n, dtype=torch.float64, device="cuda").uniform_(0.0, d, generator=g)
    y = torch.minimum(t, c)
    if ties:
        y = torch.ceil(y)
    return y.cpu().numpy(), (t <= c).to(torch.uint8).cpu().numpy()


def _lambdas(case):
    """Penalties from near the top of the path downwards: in units of the standard deviation of a null
    SNP's gradient at 0, sqrt(var x * rate / n), which puts lambda_max near 4.5."""
    sd = math.sqrt(0.35 * case["rate"] / case["n"])
    k = case["k"]
    lo = 2.5 if case.get("active") else 1.0
    f = [3.0] if k == 1 else np.exp(np.linspace(math.log(4.5), math.log(lo), k))
    return [float(v) * sd for v in f]


def _step(case):
    """1/L for near-independent columns: L = 2 ||X_c||^2 / n, ||X_c||^2 <= (sqrt n + sqrt p)^2 var x."""
    var = 1.0 if case["kind"] == "fp64_step" else 0.5
    return case["n"] / (2.0 * var * (math.sqrt(case["n"]) + math.sqrt(case["p"])) ** 2)


def _coefficients(g, case, dtype):
    """Coefficients part of the way along the fits: sparser for larger penalties."""
    k, p = case["k"], case["p"]
    b = torch.empty((k, p), dtype=dtype, device="cuda").normal_(0.0, 0.02, generator=g)
    lo = 0.005 if case.get("active") else 0.05
    share = torch.linspace(0.002, lo, k, device="cuda")[:, None]
    if case.get("active"):  # nested supports, as along one path: the union is the last column's
        u = torch.rand((1, p), device="cuda", generator=g)
    else:
        u = torch.rand((k, p), device="cuda", generator=g)
    return torch.where(u < share, b, torch.zeros_like(b))


def _make(case, seed):
    """Everything drawn from the seed: (X, time, event, beta, extras)."""
    g = _gen(seed)
    n = case["n"]
    if case["kind"] == "fp64_step":
        X = torch.empty((n, case["p"]), dtype=torch.float64, device="cuda").normal_(generator=g)
        eta = 0.3 * X[:, :20].sum(1)
        y, d = _survival(g, n, eta, case["rate"], ties=False)
        return X, y, d, _coefficients(g, case, torch.float64), None
    X = _genotypes(g, n, case["p"])
    if case["kind"] == "lipschitz":
        y, d = _survival(g, n, torch.zeros(n, dtype=torch.float64, device="cuda"), 0.2, ties=True)
        v = torch.empty(case["p"], dtype=torch.float64, device="cuda").normal_(generator=g)
        return X, y, d, None, v.cpu().numpy()
    c = _codes(X[:, :8], 32)
    c -= c.mean(0)
    eff = torch.empty(32, dtype=torch.float64, device="cuda").normal_(0.0, 0.1, generator=g)
    y, d = _survival(g, n, c @ eff, case["rate"], ties=True)
    if case["kind"] == "seq":  # sex and principal-component scores
        z = torch.empty((n, case["q"]), dtype=torch.float64, device="cuda").normal_(0.0, 0.5, generator=g)
        z[:, 0] = (z[:, 0] > 0).to(torch.float64)
        return X, y, d, None, z.cpu().numpy()
    return X, y, d, _coefficients(g, case, torch.float32), None


def _nmf_make(case, seed):
    g = _gen(seed)
    m, n, r = case["m"], case["n"], case["r"]
    X = torch.randint(0, 256, (m, n), device="cuda", generator=g, dtype=torch.int16).to(torch.float32) / 256.0
    V = torch.rand((m, r), device="cuda", generator=g)
    W = torch.rand((r, n), device="cuda", generator=g)
    return X, V, W


def prepare(case, seed):
    if case["kind"] == "nmf":
        X, V, W = _nmf_make(case, seed)
        h = NMF(X.cpu().numpy(), case["r"])
        h.set_factors(V.cpu().numpy(), W.cpu().numpy())
        return dict(case=case, h=h)
    X, y, d, beta, extra = _make(case, seed)
    if case["kind"] == "fp64_step":
        prob = CoxProblem(X.cpu().numpy(), y, d, precision="fp64")
    else:
        prob = CoxProblem(X, y, d, precision=case["precision"], p=case["p"], active_set=case.get("active", False))
    s = dict(case=case, prob=prob, beta=beta)
    if case["kind"] == "lipschitz":
        s["start"] = extra
        return s
    s["lam"] = _lambdas(case)
    s["step"] = _step(case)
    if case["kind"] == "fit":
        s["beta0"] = beta.clone()
    if case["kind"] == "autograd":
        s["beta"] = beta.requires_grad_(True)
    if case["kind"] == "seq":
        prob.set_covariates(extra)
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "nmf":
        state["h"].iterate(case["iters"], case["algo"])
        return state["h"].factors()
    prob = state["prob"]
    if kind in ("step", "fp64_step"):
        return prob.prox_step(state["beta"], state["lam"], state["step"])
    if kind == "autograd":
        state["beta"].grad = None
        loss = cox_nll(state["beta"], prob)
        loss.sum().backward()
        return loss.detach(), state["beta"].grad
    if kind == "fit":
        state["beta"].copy_(state["beta0"])
        beta, iters, obj, _ = prob.path_fit(state["lam"], state["step"], max_iter=case["iters"], tol=0.0,
                                            beta=state["beta"], warm=1)
        return beta, iters, obj
    if kind == "seq":
        B, G, iters, obj, _ = prob.path_seq(state["lam"], state["step"], max_iter=case["iters"], tol=0.0, warm=True)
        return B, G, iters, obj
    return prob.lipschitz(state["start"], tol=1e-12, maxiter=case["iters"])


def work(case):
    """Bytes: the design once per product and pass (2-bit codes, FP64 or bf16 entries), the coefficients in
    and out; flops of the products (one multiply-add per entry and column).  The active set's first product
    needs only the columns in use (0.5% of them at the start)."""
    kind = case["kind"]
    if kind == "nmf":
        m, n, r, it = case["m"], case["n"], case["r"], case["iters"]
        # V's update needs all of a row of X and W's all of V, so X is read once per iteration at least
        return dict(bytes=it * 2.0 * m * n + 8.0 * r * (m + n), flops=it * (4.0 * m * n * r + 4.0 * r * r * (m + n)))
    n, p = case["n"], case["p"]
    k = 1 if kind in ("seq", "lipschitz") else case["k"]
    x = 8.0 * n * p if kind == "fp64_step" else n * p / 4.0
    b = (16.0 if kind == "fp64_step" else 8.0) * k * p
    passes = {"fit": case.get("iters", 1), "seq": case.get("iters", 1) * case.get("k", 1),
              "lipschitz": case.get("iters", 1)}.get(kind, 1)
    first = 0.005 if case.get("active") else 1.0
    return dict(bytes=passes * (1.0 + first) * x + b, flops=passes * 2.0 * (1.0 + first) * n * p * k)


# ---- the same passes in FP64 ----------------------------------------------------------------------------

class _Design:
    """X_c = X - 1 mu^T (FP64) with rows in time order; dense in memory, or decoded block by block."""

    def __init__(self, X, p, order, center):
        self.n, self.p = X.shape[0], p
        self.X, self.order = X, order
        self.packed = X.dtype == torch.uint8
        self.rows = max(1, (1 << 28) // p)
        self.dense = None
        if not self.packed:
            self.dense = X[order]
        elif self.n * p <= 6_000_000_000:
            self.dense = torch.empty((self.n, p), dtype=torch.float64, device="cuda")
            for i, blk in self.blocks_packed():
                self.dense[i:i + blk.shape[0]] = blk
        self.mu = torch.zeros(p, dtype=torch.float64, device="cuda")
        if center:
            for _, blk in self.blocks():
                self.mu += blk.sum(0)
            self.mu /= self.n

    def blocks_packed(self):
        for i in range(0, self.n, self.rows):
            yield i, _codes(self.X[self.order[i:i + self.rows]], self.p)

    def blocks(self):
        if self.dense is not None:
            yield 0, self.dense
        else:
            yield from self.blocks_packed()

    def eta(self, B):  # (p, k) -> (n, k)
        out = torch.empty((self.n, B.shape[1]), dtype=torch.float64, device="cuda")
        for i, blk in self.blocks():
            out[i:i + blk.shape[0]] = blk @ B
        return out - (self.mu @ B)

    def xtv(self, V):  # (n, k) -> (p, k)
        out = torch.zeros((self.p, V.shape[1]), dtype=torch.float64, device="cuda")
        for i, blk in self.blocks():
            out += blk.T @ V[i:i + blk.shape[0]]
        return out - self.mu[:, None] * V.sum(0)


class _Cox:
    def __init__(self, case, X, y, d):
        y = torch.from_numpy(y).cuda()
        order = torch.argsort(y, stable=True)
        ys = y[order]
        self.order = order
        self.delta = torch.from_numpy(d).cuda()[order].to(torch.float64)[:, None]
        self.head = torch.searchsorted(ys, ys, right=False)
        self.tail = torch.searchsorted(ys, ys, right=True) - 1
        self.D = _Design(X, case["p"], order, center=case["kind"] != "fp64_step")
        self.n = len(y)

    def risk(self, eta):
        """(loss per column, delta - u): Breslow's ties."""
        c = eta.max(0).values
        w = torch.exp(eta - c)
        W = torch.flip(torch.cumsum(torch.flip(w, (0,)), 0), (0,))[self.head]
        F = torch.cumsum(self.delta / W, 0)
        loss = (self.delta * (torch.log(W) + c - eta)).sum(0) / self.n
        return loss, self.delta - w * F[self.tail]

    def step(self, B, lam, step, Z=None, gamma=None):
        """One iteration on B (p, k): (B, gamma, F of the iterate that entered)."""
        eta = self.D.eta(B)
        if Z is not None:
            eta = eta + Z @ gamma
        loss, V = self.risk(eta)
        obj = loss + lam * B.abs().sum(0)
        z = B + step * self.D.xtv(V) / self.n
        thr = step * lam
        B = torch.sign(z) * torch.clamp(z.abs() - thr, min=0.0)
        if Z is not None:
            gamma = gamma + step * (Z.T @ V) / self.n
        return B, gamma, obj


def _exact_nmf(case, seed):
    X, V, W = (t.to(torch.float64) for t in _nmf_make(case, seed))
    eps = 1e-10
    for _ in range(case["iters"]):
        if case["algo"] == "mult":
            V = V * (X @ W.T) / (V @ (W @ W.T) + eps)
            W = W * (V.T @ X) / ((V.T @ V) @ W + eps)
        else:
            G = W @ W.T
            V = torch.clamp(V - (V @ G - X @ W.T) / (2.0 * (G * G).sum() + eps), min=0.0)
            G = V.T @ V
            W = torch.clamp(W - (G @ W - V.T @ X) / (2.0 * (G * G).sum() + eps), min=0.0)
    return V, W


def exact(case, seed):
    if case["kind"] == "nmf":
        return _exact_nmf(case, seed)
    X, y, d, beta, extra = _make(case, seed)
    cox = _Cox(case, X, y, d)
    kind = case["kind"]
    if kind == "lipschitz":
        v = torch.from_numpy(extra).cuda()[:, None]
        v = v / v.norm()
        s = 0.0
        for _ in range(case["iters"]):
            b = cox.D.xtv(cox.D.eta(v))
            s = b.norm()
            v = b / s
        return 2.0 * float(s) / cox.n
    lam = torch.tensor(_lambdas(case), dtype=torch.float64, device="cuda")
    step = _step(case)
    if kind == "seq":
        Z = torch.from_numpy(extra).cuda()[cox.order]
        B = torch.zeros((case["p"], 1), dtype=torch.float64, device="cuda")
        gamma = torch.zeros((case["q"], 1), dtype=torch.float64, device="cuda")
        Bs, Gs, objs = [], [], []
        for l in range(case["k"]):
            for _ in range(case["iters"]):
                B, gamma, obj = cox.step(B, lam[l:l + 1], step, Z, gamma)
            Bs.append(B[:, 0])
            Gs.append(gamma[:, 0])
            objs.append(obj[0])
        return torch.stack(Bs), torch.stack(Gs), None, torch.stack(objs)
    B = beta.detach().to(torch.float64).T.contiguous()
    if kind == "autograd":
        loss, V = cox.risk(cox.D.eta(B))
        return loss, (-cox.D.xtv(V) / cox.n).T.contiguous()
    if kind == "fit":
        for _ in range(case["iters"]):
            B, _, obj = cox.step(B, lam, step)
        return B.T.contiguous(), None, obj
    return cox.step(B, lam, step)[0].T.contiguous()
