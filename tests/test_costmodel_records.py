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
    P.load()
    found = total = 0
    for feats, _, (form, m, n, k, budget) in RECORDS[::6]:
        es = 4 if int(form) == P.OOC_FORM_BF16X3 else 8
        cands = P.ooc_plan_candidates(int(m), int(n), int(k), es, 0, int(budget), P.make_opts(form=int(form)),
                                      capacity=64)
        F = np.array([list(c.features) for c in cands], dtype=np.float32)
        for row in feats:
            same = np.nonzero((F[:, 8:13] == row[8:13]).all(axis=1))[0]  # blocks and rings
            found, total = found + bool(len(same)), total + 1
            if len(same):
                assert np.array_equal(F[same[0], :15], row[:15])
    assert found >= 0.98 * total   # the last of 64 candidates may fall either side of the list's end
