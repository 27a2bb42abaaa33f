"""The cost model's standardisation (on the device) against numpy in FP64."""

import numpy as np
import pytest

import paper_2410_09326_gb300 as qs

pytestmark = pytest.mark.gpu


def _forward(p, x):
    f, h = qs.QS_MLP_FEATURES, qs.QS_MLP_HIDDEN
    o = 0
    for fan_out, fan_in, last in ((h, f, False), (h, h, False), (1, h, True)):
        w = p[o: o + fan_out * fan_in].reshape(fan_out, fan_in)
        b = p[o + fan_out * fan_in: o + fan_out * fan_in + fan_out]
        x = x @ w.T + b
        x = x if last else np.maximum(x, 0)
        o += fan_out * fan_in + fan_out
    return x[:, 0]


# one row, fewer and more rows than threads, more than a pass of the grid; constant features and targets, offsets
# that dwarf the spread
@pytest.mark.parametrize("n", [1, 2, 255, 257, 10007, 70000])
def test_scaling(n):
    g = np.random.default_rng(n)
    x = g.standard_normal((n, qs.QS_MLP_FEATURES)).astype(np.float32)
    x[:, 3] = 2.5
    x[:, 4] += 1000
    y = (50 + 3 * g.standard_normal(n)).astype(np.float32)
    m = qs.qs_mlp_create(1)
    try:
        before = qs.qs_mlp_params(m)
        qs.qs_mlp_train(m, x, y, epochs=1, batch=64, lr=0.0, seed=3)
        p = qs.qs_mlp_params(m)
        assert np.array_equal(p, before)
        got = qs.qs_mlp_predict(m, x)
    finally:
        qs.qs_mlp_free(m)
    xd, yd = x.astype(np.float64), y.astype(np.float64)
    sd = xd.std(0)
    sd = np.where(sd > 1e-6, sd, 1)
    ysd = yd.std() if yd.var() > 1e-12 else 1
    want = _forward(p.astype(np.float64), (xd - xd.mean(0)) / sd) * ysd + yd.mean()
    # the mean of the shifted feature is rounded to FP32 (3e-5 there); FP32 sums of 64 terms
    assert np.abs(got - want).max() <= 2e-4 * ysd + 1e-5


def test_a_model_keeps_to_its_stream():
    """On a stream that does not wait for the legacy one, every copy, memset and kernel of a model is ordered
    on that stream: its calls finish while the legacy stream is still busy, with the results of the legacy stream."""
    import torch
    g = np.random.default_rng(7)
    x = g.standard_normal((300, qs.QS_MLP_FEATURES)).astype(np.float32)
    y = g.standard_normal(300).astype(np.float32)

    def calls(m, p):
        qs.qs_mlp_params(m, p)
        grad, loss = qs.qs_mlp_gradient(m, x, y)
        qs.qs_mlp_train(m, x, y, epochs=2, batch=64, seed=3)
        return grad, loss, qs.qs_mlp_params(m), qs.qs_mlp_predict(m, x)

    side = torch.cuda.Stream()
    m, ref = qs.qs_mlp_create(1, side.cuda_stream), qs.qs_mlp_create(1)
    try:
        p = qs.qs_mlp_params(ref)
        want = calls(ref, p), calls(ref, p)  # the second continues the first's Adam moments
        got = [calls(m, p)]                  # loads the kernels and allocates
        torch.cuda.synchronize()
        busy = torch.cuda.Event()
        torch.cuda._sleep(1_000_000_000)     # about half a second
        busy.record()
        got.append(calls(m, p))
        assert not busy.query()
        for a, b in zip(want, got):
            for u, v in zip(a, b):
                assert np.array_equal(u, v)
    finally:
        torch.cuda.synchronize()
        qs.qs_mlp_free(m)
        qs.qs_mlp_free(ref)
