"""kkm_kernel_matrix in BF16 on row lengths and addresses that take the vector
and the scalar loads of the row conversion: the bits it gives for the same rows
copied to an aligned matrix and padded with zeros to a multiple of eight values
(zeros add nothing to products or norms), and for the Gaussian kernel the
values of the rounded rows in 64 bits (the kernel tolerance of the parity
tests, 1e-5 absolute)."""

import numpy as np
import pytest

from tests.helpers import KERNEL_ABS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nA,nB,d,shift", [(1, 9, 3, 0), (130, 257, 8, 0), (70, 300, 129, 0), (33, 40, 512, 1),
                                           (260, 129, 516, 0), (129, 127, 783, 3)])
@pytest.mark.parametrize("kind", ["rbf", "linear"])
def test_rows(lib, nA, nB, d, shift, kind):
    import torch
    g = torch.Generator(device="cuda").manual_seed(nA * d)
    flat = torch.rand((nA + nB) * d + shift, generator=g, device="cuda")[shift:]
    X = flat.view(nA + nB, d)  # starts `shift` floats past an aligned address
    A, B = X[:nA], X[nA:]
    sigma = 0.5 * float(np.sqrt(d))
    K = lib.kkm_kernel_matrix(A, B, kind, sigma, precision=lib.KKM_BF16)
    P = torch.zeros(nA + nB, -(-d // 8) * 8, device="cuda")
    P[:, :d] = X
    assert torch.equal(K, lib.kkm_kernel_matrix(P[:nA].contiguous(), P[nA:].contiguous(), kind, sigma,
                                                precision=lib.KKM_BF16))
    if kind == "rbf":
        a, b = A.to(torch.bfloat16).double(), B.to(torch.bfloat16).double()
        na, nb = (a * a).sum(1)[:, None], (b * b).sum(1)[None, :]
        want = torch.exp(-(na + nb - 2 * a @ b.T).clamp(min=0) / (2 * sigma * sigma))
        assert float((K.double() - want).abs().max()) <= KERNEL_ABS
