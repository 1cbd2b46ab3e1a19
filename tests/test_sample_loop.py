"""Sample-resident step loop of small networks (GPU only).

It must give the bits of the per-step kernels.  A predictor attached in
record-only mode keeps the per-step kernels without changing any arithmetic,
so both run here on the same arrays: one to four neurons per thread, several
readout warps, the largest delay, spike lists across carried windows, uneven
lengths, repeated input ids and more input events per step than the
pipelined buffers hold.
"""
from __future__ import annotations

import numpy as np
import pytest

from workloads import configs as C

pytestmark = pytest.mark.gpu


def _repeat_ids(W):
    """Doubles every step's input list (a channel listed twice spikes once)."""
    ptr, ids = W["x_ptr"], W["x_ids"]
    parts = [ids[ptr[q]:ptr[q + 1]] for q in range(len(ptr) - 1)]
    W["x_ids"] = np.concatenate([np.concatenate([p, p]) for p in parts]).astype(np.int32)
    W["x_ptr"] = 2 * ptr
    return W


CASES = {
    "one_per_thread": lambda: C.pattern_regression(T=97, n_rec=33, n_out=33),
    "two_per_thread": lambda: C.pattern_regression(T=64, n_rec=401, n_out=5, surrogate=1, reset_mode=1),
    "carried_delays": lambda: C.million_sparse(n_rec=1024, k_in=200, n_out=128, T=200, J=0.05, drive_rate=1.25,
                                               max_delay=8, lr=1e-5),
    "many_inputs": lambda: _repeat_ids(C.event_classification(
        batch=3, T=80, len_lo=41, len_hi=80, n_rec=70, side=20, events_per_300=300.0 * 300, w_in_scale=0.5,
        update_interval=40)),
    "uneven": lambda: C.event_classification(batch=5, T=75, len_lo=1, len_hi=75, n_rec=90, side=9, c_reg=1e-3,
                                             beta_reg=0.9, f_target=0.02),
}


def _run(W, per_step, mode):
    import paper_2511_21674_gb300 as ep
    s = W["spec"]
    net = ep.Network(s, W["ptr"], W["col"], W["w"], W["delay"], W["w_out"], W["out_mask"], W["feedback"],
                     record_grad=1, record_raster=1, record_psi=1, launch_mode=mode)
    pred = None
    if per_step:
        pred = ep.Predictor(s.n_out + 64, s.n_out, seed=1, max_rows=s.batch)
        net.attach_predictor(pred, mode=2)
    for _ in range(2):
        net.set_inputs(W["x_ptr"], W["x_ids"], W["targets"], W["window"], W["lengths"], s.T)
        net.simulate(s.T)
    net.sync()
    y, loss, r = net.readout(raster=True)
    out = [y, loss, r, net.surrogate(), np.asarray(net.events()), *net.weights(ep.PROJ_REC, with_grad=True),
           *net.weights(ep.PROJ_OUT, with_grad=True)]
    if s.n_in:
        out += list(net.weights(ep.PROJ_IN, with_grad=True))
    net.close()
    if pred is not None:
        pred.close()
    return out


@pytest.mark.parametrize("case", sorted(CASES))
def test_sample_loop_is_bitwise_the_per_step_kernels(case):
    W = CASES[case]()
    a, b = _run(W, True, 0), _run(W, False, 1)
    assert a[2].sum() > 0
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
