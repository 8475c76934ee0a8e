"""The network's training kernels at the edges of their tiles (128 x 64 products
over K slices of 64, vector epilogues of 16 columns, column sums of 32 columns
over 32 rows): logits, loss and gradients of one step against FP64.

Tolerance: the device rounds h1, dz2 and dz1 to BF16 (relative 2^-9 each, h1's
possibly the other way than the reference where FP32 and FP64 z1 straddle a
rounding edge), FP32 sums add 1e-6 of the sum of |terms|; worst cases, not
standard deviations, and a unit whose z lies within its error of 0 may switch."""
import numpy as np
import pytest

from oracle import quantize as Q

pytestmark = pytest.mark.gpu


def _bf16(x):
    bits = Q.f32_to_bf16_bits(np.asarray(x, np.float32))
    return bits, Q.bf16_bits_to_f32(bits).astype(np.float64)


@pytest.mark.parametrize("I,H,B", [(8, 8, 8), (72, 24, 8), (200, 136, 40), (264, 72, 136), (1024, 64, 128), (4104, 80, 264)])
def test_one_step_at_tile_edges(lib, I, H, B):
    r = np.random.default_rng(I + H + B)
    p = {"W1": r.standard_normal((I, H)) * np.sqrt(2.0 / I), "b1": r.standard_normal(H) * 0.1,
         "W2": r.standard_normal((H, H)) * np.sqrt(2.0 / H), "b2": r.standard_normal(H) * 0.1,
         "w3": r.standard_normal(H) * np.sqrt(1.0 / H), "b3": np.array([0.1])}
    p = {k: v.astype(np.float32) for k, v in p.items()}
    xb, X = _bf16(r.standard_normal((B, I)))
    y = (r.random(B) < 0.4).astype(np.float32)
    W1, W2 = _bf16(p["W1"])[1], _bf16(p["W2"])[1]
    b1, b2, w3, b3 = (p[k].astype(np.float64) for k in ("b1", "b2", "w3", "b3"))
    e = 2.0 ** -8
    z1 = X @ W1 + b1
    dz1_ = 1e-6 * (np.abs(X) @ np.abs(W1) + np.abs(b1))
    h1 = _bf16(np.maximum(z1, 0))[1]
    dh1 = e * h1 + dz1_
    z2 = h1 @ W2 + b2
    dz2_ = dh1 @ np.abs(W2) + 1e-6 * (h1 @ np.abs(W2) + np.abs(b2))
    h2 = np.maximum(z2, 0)
    s = h2 @ w3 + b3
    ds_s = dz2_ @ np.abs(w3) + 1e-6 * (h2 @ np.abs(w3) + 0.1)
    w = np.where(y > 0.5, 2.5, 1.0)
    ds = w * (1 / (1 + np.exp(-s)) - y) / B
    dds = w * 0.25 * ds_s / B + 1e-6 * np.abs(ds)
    g2 = ds[:, None] * w3
    dg2 = (dds + e * np.abs(ds))[:, None] * np.abs(w3) + np.where(np.abs(z2) <= dz2_, np.abs(g2), 0.0)
    g2 = np.where(z2 > 0, g2, 0.0)
    g1 = g2 @ W2.T
    dg1 = dg2 @ np.abs(W2).T + 1e-6 * np.abs(g2) @ np.abs(W2).T + e * np.abs(g1)
    dg1 = np.where(z1 > -dz1_, dg1, 0.0) + np.where(np.abs(z1) <= dz1_, np.abs(g1), 0.0)
    g1 = np.where(z1 > 0, g1, 0.0)
    tiny = 1e-7
    want = {"w3": (h2.T @ ds, dz2_.T @ np.abs(ds) + h2.T @ dds + 1e-6 * h2.T @ np.abs(ds)),
            "b3": (ds.sum(keepdims=True), dds.sum(keepdims=True) + 1e-6 * np.abs(ds).sum()),
            "b2": (g2.sum(0), dg2.sum(0)),
            "W2": (h1.T @ g2, dh1.T @ np.abs(g2) + h1.T @ dg2 + 1e-6 * h1.T @ np.abs(g2)),
            "b1": (g1.sum(0), dg1.sum(0)),
            "W1": (X.T @ g1, np.abs(X).T @ dg1 + 1e-6 * np.abs(X).T @ np.abs(g1))}
    m = lib.MLP(I, H, B)
    try:
        m.set_params(p)
        got_s = np.asarray(m.forward(xb), np.float64).ravel()
        assert np.all(np.abs(got_s - s) <= ds_s + tiny)
        loss = m.train_step(xb, y, 2.5, 1e-3)
        ref = np.mean(w * (np.logaddexp(0, s) - y * s))
        assert abs(loss - ref) <= np.mean(w * ds_s) + 1e-6 * abs(ref) + tiny
        got = m.get_grads()
    finally:
        m.close()
    for k, (v, t) in want.items():
        assert np.all(np.abs(np.asarray(got[k], np.float64).reshape(v.shape) - v) <= t + tiny), k
