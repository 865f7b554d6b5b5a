"""The shipped cost model, the timings it was trained on and the planner's features belong together.

costmodel_timings_gb300.npz holds the autotuner's timings of 288 problems: the shipped parameters
have the final loss of that training run on them, and the features stored with each candidate are
those that the planner computes (all but the last, the estimate, which follows the measured link).
"""
import os

import numpy as np

import paper_1808_05056_gb300 as P
from oracle import costmodel
from paper_1808_05056_gb300 import tune

RECORDS = tune.load_records(os.path.join(tune.HERE, "costmodel_timings_gb300.npz"))


def test_shipped_model_has_the_loss_of_its_training():
    X, t = tune.dataset(RECORDS)
    assert abs(costmodel.loss(tune.load().astype(np.float64), X, t) - 0.011991952) <= 1e-6


def test_features_are_the_planners():
    """Of every stored candidate that is listed with the default link rates too (the list follows the
    measured ones); each form has some."""
    P.load()
    found = {1: 0, 2: 0, 3: 0}
    for feats, _, problem in RECORDS[::6] + RECORDS[1::6] + RECORDS[2::6]:
        form, m, n, k, budget = (int(v) for v in problem)
        cands = P.ooc_plan_candidates(m, n, k, 4 if form == P.OOC_FORM_BF16X3 else 8, 0, budget,
                                      P.make_opts(form=form), capacity=64)
        F = np.array([list(c.features) for c in cands], dtype=np.float32)
        for row in feats:
            same = np.nonzero((F[:, 8:13] == row[8:13]).all(axis=1))[0]  # blocks and rings
            if len(same):
                found[form] += 1
                assert np.array_equal(F[same[0], :15], row[:15])
    assert all(found.values())
