"""Predictor kernels at the edges of their tiles (GPU only): a single row,
odd widths, several column blocks, 32-row tiles, the widest layers.  Checks
and tolerances are those of test_predictor_gpu.py (FP64 on the GPU's own BF16
operands, (K + 2) 2^-23 of the magnitude sum)."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import predictor as P
from tests.test_predictor_gpu import U23, _bf16_check, _gemm_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,n_in,H,K", [(1, 1, 16, 1), (17, 75, 33, 11), (2600, 20, 300, 5), (40, 1024, 1024, 70),
                                         (20, 1024, 1024, 1024)])
def test_train_step_at_tile_edges(R, n_in, H, K):
    import paper_2511_21674_gb300 as ep
    rng = np.random.default_rng(R)
    shapes = dict(W1=(n_in, H), b1=(H,), W2=(H, H), b2=(H,), W3=(H, K), b3=(K,))
    p = {k: (rng.standard_normal(v) / np.sqrt(v[0])).astype(np.float32) for k, v in shapes.items()}
    X = rng.standard_normal((R, n_in)).astype(np.float32)
    E = rng.standard_normal((R, K)).astype(np.float32)
    pred = ep.Predictor(n_in, K, hidden=H, params=ep.Predictor.pack(p), max_rows=R)
    loss = pred.train_step(X, E, 1e-3)
    Xb, A1, H1, A2, H2, Y = (pred.read(k) for k in ("X", "A1", "H1", "A2", "H2", "Y"))
    dY, dA2, dA1 = pred.read("dY"), pred.read("dA2"), pred.read("dA1")
    g = pred.unpack(pred.read("grads"))
    pred.close()
    Wb = {k: P.bf16(p[k]) for k in ("W1", "W2", "W3")}
    assert np.array_equal(Xb, P.bf16(X))
    _gemm_check(A1, Xb, Wb["W1"], p["b1"], "A1")
    _bf16_check(H1, P.gelu(A1), "H1")
    _gemm_check(A2, H1, Wb["W2"], p["b2"], "A2")
    _bf16_check(H2, P.gelu(A2), "H2")
    _gemm_check(Y, H2, Wb["W3"], p["b3"], "Y")
    d = Y.astype(np.float64) - E
    assert abs(loss - 0.5 * (d * d).sum() / R) <= 1e-5 * 0.5 * (d * d).sum() / R
    _bf16_check(dY, d / R, "dY", slack=2 * U23 * (np.abs(Y) + np.abs(E)) / R)
    for dA, prev, A, W, what in ((dA2, dY, A2, "W3", "dA2"), (dA1, dA2, A1, "W2", "dA1")):
        back = prev.astype(np.float64) @ Wb[W].astype(np.float64).T
        gp = P.gelu_grad(A)
        slack = (Wb[W].shape[1] + 2) * U23 * (np.abs(prev) @ np.abs(Wb[W]).T) * np.abs(gp) + 8 * U23 * np.abs(back)
        _bf16_check(dA, back * gp, what, slack=slack)
    for A, D, what in ((H2, dY, "W3"), (H1, dA2, "W2"), (Xb, dA1, "W1")):
        _gemm_check(g[what], A.T, D, None, "d" + what)
    np.testing.assert_allclose(g["b3"], (d / R).sum(0), rtol=0, atol=(R + 2) * U23 * (np.abs(d) / R).sum(0).max())
