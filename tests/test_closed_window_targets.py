"""Targets that are not finite where the learning window is closed (GPU only).

The error signal is window * (prediction - target): a NaN or infinite target
makes it NaN in every step form, also outside the window.  The sample-resident
loop skips the arithmetic there and must give what the per-step kernels (a
predictor attached in record-only mode) give.
"""
from __future__ import annotations

import numpy as np
import pytest

from workloads import configs as C

pytestmark = pytest.mark.gpu

CASES = {
    "softmax": lambda: C.event_classification(batch=3, T=60, len_lo=45, len_hi=60, n_rec=50, side=6),
    "squared": lambda: C.pattern_regression(T=70, n_rec=40, n_out=2),
    "two_warps": lambda: C.pattern_regression(T=70, n_rec=40, n_out=37),
}


def _run(W, per_step):
    import paper_2511_21674_gb300 as ep
    s = W["spec"]
    net = ep.Network(s, W["ptr"], W["col"], W["w"], W["delay"], W["w_out"], W["out_mask"], W["feedback"],
                     record_grad=1, launch_mode=0)
    pred = None
    if per_step:
        pred = ep.Predictor(s.n_out + 64, s.n_out, seed=1, max_rows=s.batch)
        net.attach_predictor(pred, mode=2)
    net.set_inputs(W["x_ptr"], W["x_ids"], W["targets"], W["window"], W["lengths"], s.T)
    net.simulate(s.T)
    out = [*net.readout(), *net.weights(ep.PROJ_IN, with_grad=True), *net.weights(ep.PROJ_REC, with_grad=True),
           *net.weights(ep.PROJ_OUT, with_grad=True)]
    net.close()
    if pred is not None:
        pred.close()
    return out


@pytest.mark.parametrize("bad", [np.nan, np.inf, 3.4e38, None])
@pytest.mark.parametrize("case", sorted(CASES))
def test_step_forms_agree_on_targets_outside_the_window(case, bad):
    W = CASES[case]()
    s = W["spec"]
    W["window"] = W["window"].copy()
    W["window"][:, :30] = 0
    W["window"][:, 40:44] = 1
    if bad is not None:
        W["targets"] = W["targets"].copy()
        W["targets"][0, 17, s.n_out - 1] = bad       # one readout at one step of the closed window
    a, b = _run(W, True), _run(W, False)
    assert np.isnan(a[1]).any() == (bad is not None and not np.isfinite(bad))
    for x, y in zip(a, b):
        assert np.array_equal(x, y, equal_nan=True)
