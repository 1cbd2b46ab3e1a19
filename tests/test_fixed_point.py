"""Fixed-point conversion of weights and back (GPU only).

One neuron that fires every step drives K readouts; the first step's readout
is the weight rounded to the 2^-32 grid (nearest even, saturated at 2^31) and
then to FP32, exactly.  Both the 32-bit conversions (magnitudes below 1, sums
below 2^16) and the 64-bit ones are reached, in the sample-resident loop and in
the per-step kernels (a predictor attached in record-only mode).
"""
from __future__ import annotations

import numpy as np
import pytest

from workloads import configs as C

pytestmark = pytest.mark.gpu

SMALL = [0.0, 2.0 ** -34, 2.0 ** -33, 3 * 2.0 ** -33, -2.0 ** -33, 2.5 * 2.0 ** -32, 1e-9, -0.3, 1 - 2.0 ** -24, -(1 - 2.0 ** -24)]
LARGE = [1.0, -1.0, 1.5, -2.7182817, 65535.996, -65536.0, 3e4, 1e9, -1e9, 3e9, -3e9]


@pytest.mark.parametrize("values", [SMALL, SMALL + LARGE], ids=["below_one", "all"])
@pytest.mark.parametrize("per_step", [False, True])
def test_readout_of_one_spike_is_the_rounded_weight(values, per_step):
    import paper_2511_21674_gb300 as ep
    w = np.asarray(values, np.float32)[None, :]
    K = w.shape[1]
    s = C.Spec(name="fixed", n_in=0, n_rec=1, n_out=K, T=1, if_period=1)
    net = ep.Network(s, np.zeros(2, np.int64), np.zeros(0, np.int32), np.zeros(0, np.float32),
                     np.zeros(0, np.uint8), w, launch_mode=0)
    if per_step:
        pred = ep.Predictor(K + 64, K, seed=1, max_rows=1)
        net.attach_predictor(pred, mode=2)
    net.set_inputs(np.zeros(2, np.int64), np.zeros(0, np.int32), np.zeros((1, 1, K), np.float32), T=1)
    net.simulate(1)
    y, _ = net.readout()
    net.close()
    # w * 2^32 is exact in FP64 (24-bit values); rint rounds to nearest even
    fx = np.clip(np.rint(w[0].astype(np.float64) * 2.0 ** 32), -2.0 ** 63, 2.0 ** 63)
    assert np.array_equal(y[0, 0], (fx * 2.0 ** -32).astype(np.float32))
