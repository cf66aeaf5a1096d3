"""Training steps of the surrogate against a plain loop over minibatches.

``train_surrogate`` takes minibatches of up to 16 tiles of 128 samples in a
kernel of its own and larger ones in a launch each.  The loop here takes each
minibatch's gradient from ``mlp_loss_grad`` and applies Adam in NumPy's FP32.
Both are sequences of IEEE operations in a fixed order (the kernels are compiled
without contraction), so the parameters agree bit for bit; the loss, a sum of
the minibatches' FP32 losses in double precision, to one unit of FP32.

Sizes: one sample; less than a tile; ragged tiles and minibatches; tiles that go
round the cluster's CTAs; the largest minibatch of the cluster kernel and the
smallest beyond it; more minibatches than one launch takes.
"""
import ctypes
import ctypes.util
import math

import numpy as np
import pytest

from oracle import mlp
from paper_2303_11811_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eng():
    import torch
    assert torch.cuda.is_available()
    from paper_2303_11811_gb300 import build, capi
    build.build()
    e = capi.Engine(32, 8, 8, 0.6)
    yield e, capi
    e.close()


@pytest.mark.parametrize("n,batch,epochs", [
    (1, 1024, 2), (100, 7, 2), (300, 128, 3), (1025, 512, 2), (5000, 1100, 2), (5001, 2048, 2),
    (5200, 2049, 2), (8500, 4097, 2), (1100, 1, 1)])
def test_steps_match_plain_loop(eng, n, batch, epochs):
    e, capi = eng
    powf = ctypes.CDLL(ctypes.util.find_library("m")).powf
    powf.restype, powf.argtypes = ctypes.c_float, [ctypes.c_float, ctypes.c_float]
    f = np.float32
    X, eps, d, r = mlp.training_samples(31, 0, n)
    X, t = X.astype(f), (eps - mlp.linear_eps(d, r)).astype(f)
    p = np.ascontiguousarray(capi.pack_mlp(inputs.mlp_init(3)), dtype=f).copy()
    e.set_mlp(p.copy())
    loss = e.train_surrogate(n, 31, epochs=epochs, batch=batch, lr=3e-3)
    m, v = np.zeros_like(p), np.zeros_like(p)
    starts = range(0, n, batch)
    total, lr, step = len(starts) * epochs, float(f(3e-3)), 0
    for _ in range(epochs):
        for b in starts:
            _, g = e.mlp_loss_grad(p, X[b:b + batch], t[b:b + batch])
            g = np.asarray(g, dtype=f)
            a = f(lr * math.pow(0.03, step / total))
            step += 1
            m = f(0.9) * m + f(0.1) * g
            v = f(0.999) * v + f(0.001) * g * g
            mh = m / (f(1) - f(powf(0.9, step)))
            vh = v / (f(1) - f(powf(0.999, step)))
            p = p - a * mh / (np.sqrt(vh) + f(1e-8))
    assert p.dtype == f
    assert np.array_equal(np.asarray(e.get_mlp(), dtype=f), p)
    want = sum(float(f(e.mlp_loss_grad(p, X[b:b + batch], t[b:b + batch])[0])) *
               len(X[b:b + batch]) for b in starts) / n
    assert abs(loss - want) <= 2.0 ** -23 * want
