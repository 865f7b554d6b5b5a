"""The planner's estimate of small launches: plans stay inside their budgets, the FP64 blocks of a
budget that holds no wave of large areas are balanced over the SMs, and short searches offer the
plan the long one (ooc_plan_candidates) ranks first."""
import math

import pytest

import paper_1808_05056_gb300 as P

SMS = 152


@pytest.fixture(scope="module", autouse=True)
def lib():
    P.build()
    P.load()


@pytest.mark.parametrize("form,es", [(P.OOC_FORM_FP64, 8), (P.OOC_FORM_OZAKI, 8), (P.OOC_FORM_BF16X3, 4)])
@pytest.mark.parametrize("M,N,K,budget", [(384, 320, 256, 1 << 20), (1024, 1024, 1024, 4 << 20),
                                          (2500, 3100, 1900, 64 << 20), (70, 5000, 333, 8 << 20),
                                          (5000, 70, 3000, 24 << 20), (12288, 12288, 12288, 288 << 20)])
def test_best_plan_fits_and_leads_the_candidates(form, es, M, N, K, budget):
    o = P.make_opts(form=form)
    try:
        p = P.ooc_plan(M, N, K, es, 1, budget, o)
    except P.OocError:
        assert form != P.OOC_FORM_FP64   # split planes may not fit the smallest budgets
        return
    assert p["device_bytes"] <= budget
    c = P.ooc_plan_candidates(M, N, K, es, 1, budget, o)[0]
    # (plans of equal estimate differ in ring sizes only in what they occupy)
    assert p["seconds"] == pytest.approx(c.est_seconds, rel=1e-12)


def test_small_fp64_blocks_are_balanced():
    p = P.ooc_plan(1024, 1024, 1024, 8, 0, 4 << 20, P.make_opts(form=P.OOC_FORM_FP64))
    tiles = math.ceil(p["mb"] / 16) * math.ceil(p["nb"] / 16)
    busiest = math.ceil(tiles / SMS)
    assert tiles / (busiest * SMS) > 0.9 and p["steps"] <= 100
