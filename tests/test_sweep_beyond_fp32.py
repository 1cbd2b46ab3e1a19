"""Adjoint sweeps whose values leave FP32's range (GPU only).

Learning signals of one sign over 50 steps take the adjoint of the filtered
eligibility past 3.4e38; an input that spiked long before reaches a finite
gradient all the same.  ALIF networks and long LIF windows, with and without
carried traces, against the eligibility recursion in 64 bits on the GPU's own
surrogate values and errors (Eq. eligibility-vector-substituted, Eq. final-
gradient); tolerance 1e-5 of the magnitude sum, as in the parity tests.
"""
from __future__ import annotations

import numpy as np
import pytest

from workloads import configs as C

pytestmark = pytest.mark.gpu

T, N = 200, 3


def _gradient(alif, state, batch, scale):
    import paper_2511_21674_gb300 as ep
    s = C.Spec(name="range", n_in=2, n_rec=N, n_out=1, T=T, batch=batch, feedback=1, lr=0.0, max_delay=3,
               neuron_model=int(alif), beta_a=1.7 if alif else 0.0, update_interval=T if state else 0)
    # channel 0: two early spikes; channel 1: every step, keeps the membranes near the threshold
    x = np.zeros((batch, T, 2), bool)
    x[:, [5, 12], 0] = True
    x[:, :, 1] = True
    col = np.tile(np.arange(N, dtype=np.int32), 2)
    net = ep.Network(s, np.array([0, N, 2 * N] + [2 * N] * N, np.int64), col,
                     np.array([0.1, 0.05, 0.12, 0.012, 0.015, 0.02], np.float32), np.array([1, 2, 3] * 2, np.uint8),
                     np.full((N, 1), 1e-3, np.float32), None, np.full((N, 1), scale, np.float32), record_grad=1,
                     record_psi=1, launch_mode=0)
    tg = np.zeros((batch, T, 1), np.float32)
    tg[:, 100:150] = -1.0
    tg[:, 180:] = 0.25
    ptr = np.concatenate([[0], np.cumsum(x.reshape(-1, 2).sum(1))]).astype(np.int64)
    net.set_inputs(ptr, np.nonzero(x.reshape(-1, 2))[1].astype(np.int32), tg, np.ones((batch, T), np.uint8),
                   np.full(batch, T, np.int32), T)
    net.simulate(T)
    y, _ = net.readout()
    psi = net.surrogate().astype(np.float64)
    _, g = net.weights(ep.PROJ_IN, with_grad=True)
    net.close()
    al, rh, ka = (np.exp(-s.dt / tau) for tau in (s.tau_m, s.tau_a, s.tau_out))
    beta = s.beta_a if alif else 0.0
    G, mag = np.zeros(N), np.zeros(N)
    for j in range(N):
        for b in range(batch):
            zb = eps = eb = pp = 0.0
            for t in range(T):
                eps = pp * zb + (rh - beta * pp) * eps
                spike = t - (j + 1) >= 0 and x[b, t - (j + 1), 0]
                zb = al * zb + float(spike)
                pp = psi[b, t, j]
                eb = ka * eb + pp * (zb - beta * eps)
                L = scale * float(y[b, t, 0] - tg[b, t, 0])
                G[j] += L * eb / batch
                mag[j] += abs(L * eb) / batch
    return g[:N], G, mag


@pytest.mark.parametrize("alif", [False, True])
@pytest.mark.parametrize("state,batch", [(False, 1), (False, 2), (True, 1), (True, 2)])
def test_adjoint_out_of_range(alif, state, batch):
    _, G, _ = _gradient(alif, state, batch, 1.0)
    scale = float(np.float32(min(6e37, 2.5e38 / (batch * np.abs(G).max()))))   # finite batch sums
    g, G, mag = _gradient(alif, state, batch, scale)
    assert np.all(np.abs(g - G) <= 1e-5 * mag)
