"""Plans of the wide form (ten e2m1 digits per coefficient), which default e4m3 handles
launch for k <= 12 and the power method always: the invariants of the two-ring pipeline
at every depth the planner accepts, the barrier protocol in the model, and which plan a
default handle launches."""
import math

import pytest

from paper_2010_16114_gb300 import _lib as L
from paper_2010_16114_gb300 import cox
from pipeline_model import random_runs


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2010_16114_gb300 import build
    build()
    return L.load()


def _check(k, p):
    cols = next(c for c in (16, 32, 64, 128) if 10 * k <= c)
    assert (p.tile_m, p.chunks, p.limb_cols) == (2, 2, cols)
    assert p.issue == 1 and p.issuers == 2 and p.mmas_per_commit == 2 * p.chunks
    G, R = p.decoder_groups, p.ring
    # one producer per ring, waits by parity: a depth of at least G + R, or a multiple of G
    assert G == 3 and R >= G and p.stages >= G + 1 and p.limb_stages >= R + 1
    for depth in (p.stages, p.limb_stages):
        assert depth >= G + R or depth % G == 0, (k, depth)
    assert p.named_barriers == math.lcm(G, R) * p.tile_m <= 15
    # 8 columns of scale factors from 504 on; accumulators and slots below them
    assert p.tmem_cols == 2 * cols + R * 4 * 16 + 8 <= 512
    kh = cols // 10
    fold = 2 * kh * 128 * 4 + 4 * kh * 4
    assert p.smem_bytes == max(120 * 1024, p.stages * 16384 + p.limb_stages * cols * 128 + 2048 + fold) <= 227 * 1024


@pytest.mark.parametrize("k", range(1, 13))
def test_every_depth_keeps_the_invariants(k):
    rc, p = L.cox_plan_form(L.COX_FORM_WIDE, k)
    assert rc == 0
    _check(k, p)
    accepted = 0
    for s in range(1, 16):
        rc, q = L.cox_plan_form(L.COX_FORM_WIDE, k, 2, 2, s, 1)
        if rc:
            assert rc == L.COX_ERR_ARG
            continue
        accepted += 1
        _check(k, q)
        assert q.stages == max(s, q.decoder_groups + 1)
    assert accepted


def test_plans_never_alias_in_the_model():
    plans = set()
    for k in range(1, 13):
        for s in range(0, 16):
            rc, p = L.cox_plan_form(L.COX_FORM_WIDE, k, 0, 0, s, 0)
            if rc == 0:
                plans.add((p.decoder_groups, p.ring, p.stages, p.limb_stages))
    assert len(plans) >= 4
    for G, R, S, S2 in sorted(plans):
        assert random_runs(G, R, S, S2, 36, runs=150, seed=11) is None, (G, R, S, S2)


def test_rejections():
    W = L.COX_FORM_WIDE
    assert L.cox_plan_form(W, 13)[0] == L.COX_ERR_ARG            # 130 digit columns
    assert L.cox_plan_form(W, 0)[0] == L.COX_ERR_ARG
    for shape in ((1, 2), (2, 1), (2, 4), (1, 4), (2, 3)):
        assert L.cox_plan_form(W, 4, *shape)[0] == L.COX_ERR_ARG  # 2 x 2 only
    for issue in (2, 3, 4):
        assert L.cox_plan_form(W, 4, 2, 2, 0, issue)[0] == L.COX_ERR_ARG
    assert L.cox_plan_form(3, 4)[0] == L.COX_ERR_ARG
    assert L.cox_plan_form(-1, 4)[0] == L.COX_ERR_ARG
    assert L.load().cox_plan_form(W, 4, 0, 0, 0, 0, None) == L.COX_ERR_ARG
    assert L.cox_plan_default(L.COX_FP64, 1)[0] == L.COX_ERR_ARG
    assert L.cox_plan_default(L.COX_SPLIT_E4M3, 65)[0] == L.COX_ERR_ARG
    assert L.cox_plan_default(L.COX_SPLIT_E2M1, 17)[0] == L.COX_ERR_ARG
    assert L.cox_plan_in_use(None, 1, 0)[0] == L.COX_ERR_ARG


def test_form_queries_agree_with_the_precision_queries():
    for prec, form in ((L.COX_SPLIT_E4M3, L.COX_FORM_E4M3), (L.COX_SPLIT_E2M1, L.COX_FORM_E2M1)):
        for k in (1, 8, 16):
            for shape in ((0, 0, 0, 0), (2, 2, 0, 1)):
                a, b = L.cox_plan_shape_prec(prec, k, *shape), L.cox_plan_form(form, k, *shape)
                assert a[0] == b[0] == 0
                assert all(getattr(a[1], f) == getattr(b[1], f) for f, _ in L.cox_plan._fields_)


@pytest.mark.parametrize("k", range(1, 65))
def test_default_plans(k):
    d = cox.default_plan(k)
    if k <= 12:
        assert d["form"] == "wide" and (d["tile_m"], d["chunks"]) == (2, 2)
    else:
        want = (2, 2, 3) if k <= 16 else (2, 2, 2) if k <= 32 else (1, 1, 3)
        assert d["form"] == "e4m3" and (d["tile_m"], d["chunks"], d["decoder_groups"]) == want
        assert d["limb_cols"] >= 4 * k
    if k <= 16:
        e = cox.default_plan(k, "split_e2m1")
        assert e["form"] == "e2m1" and (e["tile_m"], e["chunks"]) == (2, 2)
