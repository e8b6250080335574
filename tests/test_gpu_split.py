"""The FP32 Gaussian block on the tensor cores (three 9-bit slices per value)
against 64-bit values.

Tolerance per entry, derived: the norms and the dot product are FP32 roundings
of sums of size |a|^2 + |b|^2 (at most 4 + 4 units of 2^-24 of it), so K =
exp(-d2 / (2 sigma^2)) is off by at most 8 * 2^-24 (|a|^2 + |b|^2) / (2 sigma^2)
plus the exponential's own 2^-21.  Sizes: one entry past and short of the
128 x 256 and 128 x 64 tiles, row lengths off the 32-value stage and the
256-value chunk, the shortest rows that take this path."""

import numpy as np
import pytest

from synth import blobs, mnist_like

pytestmark = pytest.mark.gpu


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x, np.float32)).to("cuda:0")


def _check(K, A, B, sigma):
    a, b = A.astype(np.float64), B.astype(np.float64)
    na, nb = (a * a).sum(1)[:, None], (b * b).sum(1)[None, :]
    d2 = np.maximum(na + nb - 2.0 * a @ b.T, 0.0)
    tol = 2.0 ** -21 + 8 * 2.0 ** -24 * (na + nb) / (2 * sigma * sigma)
    off = np.abs(K - np.exp(-d2 / (2 * sigma * sigma)))
    assert np.all(off <= tol), float(np.max(off / tol))


@pytest.mark.parametrize("nA,nB,d", [(33, 1, 64), (257, 129, 65), (255, 127, 100), (64, 128, 256), (65, 700, 257),
                                     (300, 9800, 784), (1025, 20001, 96), (256, 19456, 513)])
@pytest.mark.parametrize("data", ["features", "far"])
def test_matrix_against_64_bits(lib, nA, nB, d, data):
    if data == "features":
        X, _ = mnist_like(nA + nB, d, 5, problem=nA + d)
        sigma = 0.3 * np.sqrt(d)
    else:
        X, _ = blobs(nA + nB, d, 4, problem=nA + d)
        X = X + np.float32(40.0)
        sigma = 6.0 * np.sqrt(d)
    K = lib.kkm_kernel_matrix(_dev(X[:nA]), _dev(X[nA:]), "rbf", sigma).cpu().numpy()
    _check(K, X[:nA], X[nA:], float(np.float32(sigma)))


def test_scales_and_non_finite_rows(lib):
    """Rows far apart in magnitude, zero and subnormal rows; a row with NaN or
    Inf gives what the FFMA kernel gives (its other rows keep their values)."""
    g = np.random.default_rng(5)
    X = g.normal(size=(400, 80)).astype(np.float32)
    X[::7] *= np.float32(2.0 ** -70)
    X[3::7] *= np.float32(2.0 ** 9)
    X[5] = 0.0
    X[12] = np.float32(1e-42)
    A, B = X[:150], X[150:]
    K = lib.kkm_kernel_matrix(_dev(A), _dev(B), "rbf", 300.0).cpu().numpy()
    _check(K, A, B, 300.0)
    B = B.copy()
    B[17, 3] = np.nan
    B[40, 0] = np.inf
    got = lib.kkm_kernel_matrix(_dev(A), _dev(B), "rbf", 300.0).cpu().numpy()
    keep = np.setdiff1d(np.arange(len(B)), [17, 40])
    _check(got[:, keep], A, B[keep], 300.0)
    assert np.all(got[:, 17] == 1.0) and np.all((got[:, 40] == 0.0) | (got[:, 40] == 1.0))


@pytest.mark.parametrize("mode,C", [("supports", 6), ("medoids", 40)])
def test_assign_does_not_depend_on_the_other_rows(lib, mode, C):
    X, _ = mnist_like(9000, 150, 10, problem=3)
    S, Q = _dev(X[:700]), _dev(X[700:])
    _, model = lib.kkm_fit(S, C, 1, 1.0, "rbf", 3.0, iters=2, seed=1)
    lab, dist = lib.kkm_assign(model, Q, mode)
    for rows in ([0], list(range(130)), list(range(4000, 8300))):
        la, da = lib.kkm_assign(model, Q[rows].contiguous(), mode)
        assert np.array_equal(la.cpu().numpy(), lab[rows].cpu().numpy())
        assert np.array_equal(da.cpu().numpy(), dist[rows].cpu().numpy())


@pytest.mark.parametrize("mode", ["supports", "medoids"])
def test_assign_of_non_finite_rows_writes_nothing(lib, mode):
    import ctypes
    import torch
    X, _ = mnist_like(1200, 90, 4, problem=4)
    _, model = lib.kkm_fit(_dev(X[:600]), 4, 1, 1.0, "rbf", 2.0, iters=2, seed=1)
    Q = _dev(X[600:])
    Q[5, 7] = float("inf")
    lab = torch.full((600,), -7, dtype=torch.int32, device="cuda:0")
    dist = torch.full((600,), -7.0, device="cuda:0")
    rc = lib.load().kkm_assign(model.handle, ctypes.c_void_p(Q.data_ptr()), 600, lib.MODE[mode],
                               ctypes.c_void_p(lab.data_ptr()), ctypes.c_void_p(dist.data_ptr()), None)
    assert rc == lib.STATUS_EINVAL and bool((lab == -7).all()) and bool((dist == -7.0).all())
