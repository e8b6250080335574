"""K(A, A) is symmetric to the last bit on every kernel block: FFMA, FP16 slices
(from tile edges to several tiles a side, with rows they do not hold), BF16, FP8
and MD frames; from device memory, from the host and from a strided view."""

import numpy as np
import pytest

from synth import md_trajectory, mnist_like

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,prec", [(33, 130, "fp32"), (129, 128, "fp32"), (257, 784, "fp32"), (1500, 784, "fp32"),
                                      (3001, 200, "fp32"), (200, 40, "fp32"), (700, 300, "bf16"), (700, 300, "fp8")])
def test_rbf(lib, n, d, prec):
    import torch
    X, _ = mnist_like(n, d, 5, problem=n)
    X[n // 2] *= np.float32(0.001)
    X[n // 2, 3] = 2.0
    p = {"fp32": lib.KKM_FP32, "bf16": lib.KKM_BF16, "fp8": lib.KKM_FP8}[prec]
    sigma = 0.3 * np.sqrt(d)
    A = torch.from_numpy(np.ascontiguousarray(X, np.float32)).to("cuda:0")
    K = lib.kkm_kernel_matrix(A, A, "rbf", sigma, precision=p)
    assert torch.equal(K, K.T)
    wide = torch.zeros(n, d + 3, device="cuda:0")
    wide[:, :d] = A
    view = wide[:, :d]
    assert torch.equal(lib.kkm_kernel_matrix(view, view, "rbf", sigma, precision=p), K)
    host = np.ascontiguousarray(X, np.float32)
    assert np.array_equal(lib.kkm_kernel_matrix(host, host, "rbf", sigma, precision=p), K.cpu().numpy())
    # one row set of another buffer: the same values up to the order of two sums
    other = lib.kkm_kernel_matrix(A, A.clone(), "rbf", sigma, precision=p)
    assert torch.equal(torch.triu(other), torch.triu(K)) and float((other - K).abs().max()) <= 2.0 ** -21


def test_frames(lib):
    import torch
    F, _ = md_trajectory(n_frames=300, n_atoms=40, n_states=3, dwell=50.0, workload=84)
    A = torch.from_numpy(np.ascontiguousarray(F.reshape(300, -1), np.float32)).to("cuda:0")
    K = lib.kkm_kernel_matrix(A, A, "rmsd", 1.5, 40)
    assert float((K - K.T).abs().max()) <= 1e-5
