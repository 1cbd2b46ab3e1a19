"""Batch sums whose partial values leave FP32's range (GPU only).

The batched gradients add a synapse's terms as FP32 pairs.  Terms of either
sign whose running sum passes 3.4e38 must still give the sum (as an FP64 sum
does), and sums beyond FP32 the infinity of their sign, in the single-window
form (sum over arrivals) and in the windowed form (sum over samples).  The
reference is the eligibility recursion in 64 bits on the GPU's own surrogate
values and errors; FP32 terms, so 1e-5 of the magnitude sum.
"""
from __future__ import annotations

import numpy as np
import pytest
from scipy.signal import lfilter

from workloads import configs as C

pytestmark = pytest.mark.gpu

T, N, D = 60, 3, (1, 2, 4)


def _run(n_syn, targets, scale, U):
    """n_syn synapses per input row (short rows are split over threads)."""
    import paper_2511_21674_gb300 as ep
    B = len(targets)
    s = C.Spec(name="range", n_in=1, n_rec=n_syn, n_out=1, T=T, batch=B, feedback=1, lr=0.0, max_delay=max(D),
               update_interval=U)
    x = np.tile(np.arange(T) % 5 == 2, (B, 1))
    fb = np.full((n_syn, 1), scale, np.float32)
    delay = np.array([D[j % 3] for j in range(n_syn)], np.uint8)
    net = ep.Network(s, np.concatenate([[0], np.full(n_syn + 1, n_syn)]).astype(np.int64),
                     np.arange(n_syn, dtype=np.int32), np.full(n_syn, 0.05, np.float32), delay,
                     np.full((n_syn, 1), 1e-3, np.float32), None, fb, record_grad=1, record_psi=1, launch_mode=0)
    tg = np.broadcast_to(np.asarray(targets, np.float32)[:, None, None], (B, T, 1)).copy()
    net.set_inputs(np.concatenate([[0], np.cumsum(x.ravel())]).astype(np.int64), np.zeros(int(x.sum()), np.int32),
                   tg, np.ones((B, T), np.uint8), np.full(B, T, np.int32), T)
    net.simulate(T)
    y, _ = net.readout()
    psi = net.surrogate().astype(np.float64)
    _, g = net.weights(ep.PROJ_IN, with_grad=True)
    net.close()
    alpha, kappa = np.exp(-s.dt / s.tau_m), np.exp(-s.dt / s.tau_out)
    G, mag = np.zeros((2, B, n_syn))
    for j in range(n_syn):
        d = int(delay[j])
        z = np.concatenate([np.zeros(d), x[0, :-d]]).astype(np.float64)
        for b in range(B):
            L = float(fb[j, 0]) * (y[b, :, 0].astype(np.float64) - tg[b, :, 0])
            ebar = lfilter([1.0], [1.0, -kappa], psi[b, :, j] * lfilter([1.0], [1.0, -alpha], z))
            G[b, j], mag[b, j] = L @ ebar, np.abs(L) @ np.abs(ebar)
    return g, G, mag


@pytest.mark.parametrize("n_syn", [3, 300])
@pytest.mark.parametrize("U", [0, 30, 60])
def test_partial_sums_out_of_range(U, n_syn):
    targets = [-1.0, -1.0, -1.0, 1.0, 1.0, 0.75]     # each sample below the range, three of them above
    _, G, _ = _run(n_syn, targets, 1.0, U)
    scale = 2e38 / np.abs(G).max()
    g, G, mag = _run(n_syn, targets, scale, U)
    B = len(targets)
    assert np.abs(G).max() < 3.4e38 and np.abs(np.cumsum(G, 0)).max() > 3.5e38
    assert np.abs(G.sum(0)).max() < 3.3e38
    assert np.all(np.abs(g - G.sum(0) / B) <= 1e-5 * mag.sum(0) / B)


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("U", [0, 60])
def test_sums_out_of_range_are_infinite(U, sign):
    _, G, _ = _run(3, [-1.0] * 8, 1.0, U)
    g, G, _ = _run(3, [-sign] * 8, 2e38 / np.abs(G).max(), U)
    assert np.abs(G.sum(0)).min() > 3.5e38
    assert np.array_equal(g, sign * np.full(3, np.inf, np.float32))
