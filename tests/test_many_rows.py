"""Batched gradients of networks with many short rows (GPU only).

From some thousand source rows on, the batched kernels give a row to a warp.
Checked against the oracle with few and many samples, with rows whose spikes
exceed the warp's list (neurons that fire on a schedule), in the single-window
and in the windowed form.
"""
from __future__ import annotations

import pytest

from tests.test_gpu_parity import run_parity
from workloads import configs as C

pytestmark = pytest.mark.gpu


def _net(batch, T, U, **over):
    # 8000 rows: above 48 per SM
    return C.million_sparse(n_rec=8000, k_in=3, n_out=2, T=T, J=0.3, lr=1e-5, batch=batch, continuous=0,
                            update_interval=U, **over)


@pytest.mark.parametrize("batch,T,over", [(1, 40, {}), (2, 40, {}), (30, 37, dict(if_period=1))])
def test_single_window(batch, T, over):
    rep = run_parity(_net(batch, T, 0, **over), gpu_kw=dict(trace_kernel=2))
    assert rep["spikes"] > 1000


@pytest.mark.parametrize("batch,over", [(2, {}), (40, dict(if_period=2)), (3, dict(neuron_model=1, beta_a=1.7))])
def test_windows(batch, over):
    rep = run_parity(_net(batch, 40, 20, **over))
    assert rep["spikes"] > 1000
