"""Rows whose coordinates spread: the FP32 Gaussian block on the tensor cores
holds a row's values below its largest one, and its error against 64 bits must
be no larger than that of an FP32 FFMA product.

The yardstick is that product itself, emulated here: sums of 32 products, one
FP32 rounding each (the exact product of two FP32 values fits FP64), added in
FP32, then the same norms and clamp.  The bandwidth puts exponents near -15, so
that log K gives the squared distance back to 2^-24 of itself; both are read
through the factor -log2(e) / (2 sigma^2) as the kernels round it.  Tolerance: the
products the slices leave out, 0.23 sqrt(2 d) in units of the row scale, come to
at most a third of the FFMA error for the widest rows here, which in quadrature
is 1.06 of it; 1.1 leaves the rest to the spread of a mean over 100,000 pairs."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _rows(name, n, d, g):
    if name.startswith("lognormal"):
        return np.exp(float(name[9:]) * g.normal(size=(n, d)))
    flat = name.startswith("flat")
    x = 0.25 + 0.002 * g.normal(size=(n, d)) if flat else g.uniform(0.1, 0.4, size=(n, d))
    x[np.arange(n), g.integers(0, d, n)] = float(name.lstrip("flatspike"))
    return x


def _ffma_sq_dist(A, B):
    dot = np.zeros((len(A), len(B)), np.float32)
    for c0 in range(0, A.shape[1], 32):
        part = np.zeros_like(dot)
        for c in range(c0, min(c0 + 32, A.shape[1])):
            part = (part.astype(np.float64) + np.multiply.outer(A[:, c].astype(np.float64), B[:, c])).astype(np.float32)
        dot += part
    na = (A.astype(np.float64) ** 2).sum(1).astype(np.float32)
    nb = (B.astype(np.float64) ** 2).sum(1).astype(np.float32)
    return np.maximum((na[:, None] + nb[None, :]) - 2 * dot, np.float32(0))


@pytest.mark.parametrize("name,d", [("spike4", 64), ("spike8", 256), ("spike8", 784), ("spike30", 784), ("flat30", 784),
                                    ("flat8", 130), ("lognormal1", 784), ("lognormal1.5", 300), ("lognormal2", 784),
                                    ("lognormal2", 2048)])
def test_error_no_larger_than_ffma(lib, name, d):
    import torch
    g = np.random.default_rng(d)
    n = 1024 if d < 96 else 256
    X = _rows(name, n + 400, d, g).astype(np.float32)
    A, B = X[:n], X[n:]
    a, b = A.astype(np.float64), B.astype(np.float64)
    norms = (a * a).sum(1)[:, None] + (b * b).sum(1)[None, :]
    d2 = np.maximum(norms - 2 * a @ b.T, 0)
    sigma = np.float32(np.sqrt(np.median(d2) / 30))
    factor = np.float32(-1.4426950408889634 / (2 * float(sigma) ** 2))
    K = lib.kkm_kernel_matrix(torch.from_numpy(A).to("cuda:0"), torch.from_numpy(B).to("cuda:0"), "rbf", float(sigma))
    K = K.cpu().numpy().astype(np.float64)
    seen = K > 1e-30
    ffma = (_ffma_sq_dist(A, B) * factor).astype(np.float64) / float(factor)

    def rms(v):
        return np.sqrt(np.mean((((v - d2) / norms)[seen] * 2.0 ** 24) ** 2))

    got, want = rms(np.log2(np.maximum(K, 1e-300)) / float(factor)), rms(ffma)
    assert seen.mean() > 0.4 and got <= 1.1 * want, (got, want)
