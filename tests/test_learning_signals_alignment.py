"""Learning-signal product on feedback rows that are not 16-byte aligned (GPU
only): the vector and the scalar producers give the same bits."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_rec,U,K", [(1000, 100, 100), (129, 17, 4), (300, 128, 128)])
def test_unaligned_feedback_gives_the_same_bits(n_rec, U, K):
    import torch
    import paper_2511_21674_gb300 as ep
    g = torch.Generator(device="cuda").manual_seed(n_rec)
    flat = torch.randn(n_rec * K + 1, generator=g, device="cuda")
    E = torch.randn(1, U, K, generator=g, device="cuda")
    shifted = flat[1:].view(n_rec, K)
    assert shifted.data_ptr() % 16 != 0
    assert torch.equal(ep.learning_signals(shifted, E), ep.learning_signals(shifted.clone(), E))
