"""Predictor kernels where the tile's buffers or the ring's stages differ
(GPU only): hidden widths with and without padding columns (the second layer's
output takes the inputs' place or not), inputs wider and narrower than the
hidden layers, narrow networks over several waves of tiles, one full and one
ragged column block, infinite inputs beside a layer whose tile they share.
Checks and tolerances are those of test_predictor_gpu.py."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import predictor as P
from tests.test_predictor_gpu import U23, _bf16_check, _gemm_check

pytestmark = pytest.mark.gpu


def _params(rng, n_in, H, K):
    shapes = dict(W1=(n_in, H), b1=(H,), W2=(H, H), b2=(H,), W3=(H, K), b3=(K,))
    return {k: (rng.standard_normal(v) / np.sqrt(v[0])).astype(np.float32) for k, v in shapes.items()}


@pytest.mark.parametrize("R,n_in,H,K", [(5000, 74, 16, 10), (10_000, 90, 40, 3), (5000, 3, 64, 70), (40, 900, 48, 260),
                                         (33, 30, 272, 1), (700, 600, 600, 300), (5000, 74, 256, 10)])
def test_train_step_of_other_shapes(R, n_in, H, K):
    import paper_2511_21674_gb300 as ep
    rng = np.random.default_rng(R + H)
    p = _params(rng, n_in, H, K)
    X = rng.standard_normal((R, n_in)).astype(np.float32)
    E = rng.standard_normal((R, K)).astype(np.float32)
    pred = ep.Predictor(n_in, K, hidden=H, params=ep.Predictor.pack(p), max_rows=R)
    Yf = pred.forward(X)
    pred.train_step(X, E, 1e-3)
    Xb, A1, H1, A2, H2, Y = (pred.read(k) for k in ("X", "A1", "H1", "A2", "H2", "Y"))
    dY, dA2, dA1 = pred.read("dY"), pred.read("dA2"), pred.read("dA1")
    g = pred.unpack(pred.read("grads"))
    pred.close()
    Wb = {k: P.bf16(p[k]) for k in ("W1", "W2", "W3")}
    assert np.array_equal(Xb, P.bf16(X)) and np.array_equal(Yf, Y)
    _gemm_check(A1, Xb, Wb["W1"], p["b1"], "A1")
    _bf16_check(H1, P.gelu(A1), "H1")
    _gemm_check(A2, H1, Wb["W2"], p["b2"], "A2")
    _bf16_check(H2, P.gelu(A2), "H2")
    _gemm_check(Y, H2, Wb["W3"], p["b3"], "Y")
    d = Y.astype(np.float64) - E
    _bf16_check(dY, d / R, "dY", slack=2 * U23 * (np.abs(Y) + np.abs(E)) / R)
    for dA, prev, A, W, what in ((dA2, dY, A2, "W3", "dA2"), (dA1, dA2, A1, "W2", "dA1")):
        back = prev.astype(np.float64) @ Wb[W].astype(np.float64).T
        gp = P.gelu_grad(A)
        slack = (Wb[W].shape[1] + 2) * U23 * (np.abs(prev) @ np.abs(Wb[W]).T) * np.abs(gp) + 8 * U23 * np.abs(back)
        _bf16_check(dA, back * gp, what, slack=slack)
    for A, D, what in ((H2, dY, "W3"), (H1, dA2, "W2"), (Xb, dA1, "W1")):
        _gemm_check(g[what], A.T, D, None, "d" + what)


@pytest.mark.parametrize("n_in,H", [(30, 48), (100, 40), (100, 48)])
def test_rows_do_not_see_one_another(n_in, H):
    """A row of infinities leaves the other rows' outputs as they are."""
    import paper_2511_21674_gb300 as ep
    rng = np.random.default_rng(1)
    pred = ep.Predictor(n_in, 5, hidden=H, params=ep.Predictor.pack(_params(rng, n_in, H, 5)), max_rows=20)
    X = rng.standard_normal((20, n_in)).astype(np.float32)
    want = pred.forward(X)
    X[7] = np.inf
    got = pred.forward(X)
    pred.close()
    keep = np.arange(20) != 7
    assert np.array_equal(got[keep], want[keep])
