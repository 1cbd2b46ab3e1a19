"""Inputs refused after earlier ones were accepted (GPU only).

A refusal that comes once the earlier inputs are overwritten (device arrays are
checked after the copy) or their window buffers given back (a window too long
for the band-major form) leaves nothing to simulate: the next simulate call is
refused instead of running on what is left, and new inputs are accepted.  A
refusal of host arrays comes before anything is touched.
"""
from __future__ import annotations

import numpy as np
import pytest

from workloads import configs as C

pytestmark = pytest.mark.gpu


def _dev(W, ids):
    import torch
    return [torch.as_tensor(np.ascontiguousarray(a)).cuda() for a in
            (W["x_ptr"], ids.astype(np.int32), W["targets"], W["window"], W["lengths"])]


def test_device_inputs_with_a_bad_channel():
    import paper_2511_21674_gb300 as ep
    W = C.pattern_regression(T=50, n_rec=30)
    s = W["spec"]
    net = ep.Network(s, W["ptr"], W["col"], W["w"], W["delay"], W["w_out"], launch_mode=0)
    net.set_inputs(*_dev(W, W["x_ids"]), T=50)
    net.simulate(50)
    bad = W["x_ids"].copy()
    bad[-1] = s.n_in
    with pytest.raises(ep.EpropError, match="input id"):
        net.set_inputs(*_dev(W, bad), T=50)
    with pytest.raises(ep.EpropError, match="must come first"):
        net.simulate(50)
    # host arrays are looked at before anything is copied: the accepted inputs stay
    net.set_inputs(W["x_ptr"], W["x_ids"], W["targets"], W["window"], W["lengths"], 50)
    with pytest.raises(ep.EpropError, match="input id"):
        net.set_inputs(W["x_ptr"], bad, W["targets"], W["window"], W["lengths"], 50)
    net.simulate(50)
    net.sync()
    net.close()


def test_shorter_device_inputs_refused_between_longer_ones():
    import paper_2511_21674_gb300 as ep
    W, S = C.pattern_regression(T=90, n_rec=30), C.pattern_regression(T=40, n_rec=30)
    s = W["spec"]
    net = ep.Network(s, W["ptr"], W["col"], W["w"], W["delay"], W["w_out"], launch_mode=1, record_raster=1)
    net.set_inputs(*_dev(W, W["x_ids"]), T=90)
    net.simulate(90)
    want = net.readout(raster=True)
    bad = S["x_ids"].copy()
    bad[0] = -1
    with pytest.raises(ep.EpropError, match="input id"):
        net.set_inputs(*_dev(S, bad), T=40)
    for call in (net.readout, lambda: net.simulate(90), lambda: net.simulate(40)):
        with pytest.raises(ep.EpropError):
            call()
    net.set_inputs(*_dev(W, W["x_ids"]), T=90)
    net.simulate(90)
    got = net.readout(raster=True)
    net.close()
    assert got[0].shape == want[0].shape and np.isfinite(got[0]).all() and got[2].sum() > 0


def test_window_too_long_for_the_band_form():
    import paper_2511_21674_gb300 as ep
    W = C.million_sparse(n_rec=200, k_in=20, n_out=1, T=40, J=0.05, update_interval=0)
    s = W["spec"]
    net = ep.Network(s, W["ptr"], W["col"], W["w"], W["delay"], W["w_out"], None, W["feedback"], launch_mode=0,
                     trace_kernel=4)
    x_ids = np.zeros(0, np.int32)
    net.set_inputs(W["x_ptr"], x_ids, W["targets"], T=40)
    T = 70_000
    with pytest.raises(ep.EpropError, match="update windows"):
        net.set_inputs(np.zeros(T + 1, np.int64), x_ids, np.zeros((1, T, 1), np.float32), T=T)
    with pytest.raises(ep.EpropError, match="must come first"):
        net.simulate(40)
    net.set_inputs(W["x_ptr"], x_ids, W["targets"], T=40)
    net.simulate(40)
    net.sync()
    net.close()
