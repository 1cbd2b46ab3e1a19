"""The cooperative step loop (launch_mode 2) on networks beyond the sample
loop's sizes (GPU only).

Networks of up to 1024 recurrent neurons run in the sample-resident loop in every
launch mode; larger ones run their steps in one cooperative kernel with grid
barriers in launch_mode 2 and in per-step launches in modes 0 and 1.  All three
must give the same bits, for one sample and for a batch of uneven lengths with
input channels, drive and delays; the batch is also checked against the FP64
oracle in both forms (the parity rules of test_gpu_parity.py).
"""
from __future__ import annotations

import numpy as np
import pytest

from tests.test_gpu_parity import _gpu_net, run_parity
from workloads import configs as C

pytestmark = pytest.mark.gpu

CASES = {
    # adaptive neurons, input events inside the neuron kernel, softmax
    "batch_alif": lambda: C.event_classification(batch=3, T=70, len_lo=1, len_hi=70, n_rec=1100, side=8,
                                                 events_per_300=3000.0),
    # two thousand neurons, delays, drive, fixed feedback, one sample and two
    "single_delays": lambda: C.million_sparse(n_rec=2000, k_in=60, n_out=3, T=80, J=0.05, lr=1e-5, continuous=0,
                                              update_interval=0),
    "batch_delays": lambda: C.million_sparse(n_rec=1500, k_in=60, n_out=130, T=60, J=0.05, lr=1e-5, continuous=0,
                                             update_interval=0, batch=2),
    # the compiled-in variants: fixed reset, exponential surrogate, rate regularisation
    "variants": lambda: C.pattern_regression(T=60, n_rec=1030, n_out=2, surrogate=1, reset_mode=1, c_reg=1e-3,
                                             beta_reg=0.9, f_target=0.02),
}


def _outputs(W, mode):
    import paper_2511_21674_gb300 as ep
    s = W["spec"]
    net = _gpu_net(W, launch_mode=mode)
    for _ in range(2):
        net.set_inputs(W["x_ptr"], W["x_ids"], W["targets"], W["window"], W["lengths"], s.T)
        net.simulate(s.T)
    net.sync()
    y, loss, r = net.readout(raster=True)
    launches = net.stats()["kernel_launches"]
    out = [y, loss, r, net.surrogate(), np.asarray(net.events()), *net.weights(ep.PROJ_REC, with_grad=True),
           *net.weights(ep.PROJ_OUT, with_grad=True)]
    if s.n_in:
        out += list(net.weights(ep.PROJ_IN, with_grad=True))
    net.close()
    return out, launches


@pytest.mark.parametrize("case", sorted(CASES))
def test_one_launch_is_bitwise_the_per_step_launches(case):
    W = CASES[case]()
    eager, l0 = _outputs(W, 0)
    graph, l1 = _outputs(W, 1)
    loop, l2 = _outputs(W, 2)
    # per-step launches in modes 0 and 1, one launch for all steps in mode 2
    assert l0 == l1 >= 2 * W["spec"].T and l2 < 20
    assert eager[2].sum() > 0
    for x, y, z in zip(eager, graph, loop):
        assert np.array_equal(x, y) and np.array_equal(x, z)


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("case", ["batch_alif", "batch_delays"])
def test_large_batches_against_the_oracle(case, mode):
    rep = run_parity(CASES[case](), gpu_kw=dict(launch_mode=mode))
    assert rep["spikes"] > 100
