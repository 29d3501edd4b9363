"""Cost-model gradients, predictions and one training step at the edges of the
fused row kernel (8 rows a CTA, at most 256 hidden units in steps of 8) and of
the gradient kernel's row splits, and on widths that run layer by layer.  The
oracle gets the BF16-rounded weights in FP64; what is left is FP32 arithmetic
over sums of at most 4097 terms: 1e-4 relative per gradient tensor.
"""
import numpy as np
import pytest

from oracle import mlp as omlp

pytestmark = pytest.mark.gpu

D = 16


@pytest.mark.parametrize("hidden,n", [(8, 1), (64, 9), (72, 65), (256, 7), (256, 1000), (256, 4097), (20, 33), (264, 40)])
def test_gradients_and_predictions(hidden, n):
    from paper_2104_10523_gb300 import build, tnq as T
    build.build()
    ctx = T.Context(0, "fp32")
    m = T.CostModel(ctx, hidden=hidden, max_batch=4100, seed=3)
    P = omlp.init_params(D, hidden, seed=hidden)
    rng = np.random.default_rng(n)
    for k in ("b1", "b2", "b3"):
        P[k] = rng.standard_normal(P[k].shape) * 0.1
    m.set_params(np.concatenate([P[k].reshape(-1) for k in omlp.PARAMS]))
    for k in P:
        P[k] = np.asarray(P[k], np.float32).astype(np.float64)
    for k in ("W1", "W2", "W3"):
        P[k] = omlp.bf16_round(P[k])
    X = rng.uniform(0, 1, size=(n, D)).astype(np.float32)
    t = rng.standard_normal(n).astype(np.float32)
    g, loss = m.gradients(X, t)
    G = omlp.gradients(P, X.astype(np.float64), t.astype(np.float64))
    at = 0
    for k in omlp.PARAMS:
        got = g[at:at + G[k].size].reshape(G[k].shape)
        at += G[k].size
        assert np.linalg.norm(got - G[k]) <= 1e-4 * np.linalg.norm(G[k]), k
    ref = omlp.loss(P, X.astype(np.float64), t.astype(np.float64))
    assert abs(loss - ref) <= 1e-5 * ref
    y, _ = omlp.forward(P, X.astype(np.float64))
    assert np.linalg.norm(m.predict(X) - y) <= 1e-5 * np.linalg.norm(y)
    # the parameters move and their BF16 copies with them: the loss falls
    m.train(X, t, epochs=30, batch=min(n, 1024), lr=1e-3)
    assert m.gradients(X, t)[1] < loss
