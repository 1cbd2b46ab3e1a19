"""Error filter with many (sample, readout) pairs (GPU only).

From some ten thousand pairs on one thread filters a pair's error over the
window instead of a warp; readout weights and gradients against the oracle,
with a window that its batches of steps do not divide.
"""
from __future__ import annotations

import pytest

from tests.test_gpu_parity import run_parity
from workloads import configs as C

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("U", [0, 19])
def test_many_readouts_and_samples(U):
    # 20 x 512 = 10,240 pairs: above 64 per SM
    W = C.million_sparse(n_rec=60, k_in=5, n_out=512, T=38, J=0.3, lr=1e-5, batch=20, continuous=0, update_interval=U,
                         drive_rate=2.0)
    rep = run_parity(W)
    assert rep["spikes"] > 100
