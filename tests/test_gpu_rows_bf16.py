"""kkm_kernel_matrix in BF16 on row lengths and addresses that take the vector
and the scalar loads of the row conversion, against the kernel of the rounded
rows in 64 bits (the kernel tolerance of the parity tests, 1e-5 absolute; for
the linear kernel 2^-20 of |a| |b|, FP32 accumulation)."""

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
    K = lib.kkm_kernel_matrix(A, B, kind, sigma, precision=lib.KKM_BF16).double()
    a, b = A.to(torch.bfloat16).double(), B.to(torch.bfloat16).double()
    dot = a @ b.T
    na, nb = (a * a).sum(1)[:, None], (b * b).sum(1)[None, :]
    if kind == "linear":
        assert bool(((K - dot).abs() <= 2.0 ** -20 * (na * nb).sqrt()).all())
    else:
        want = torch.exp(-(na + nb - 2 * dot).clamp(min=0) / (2 * sigma * sigma))
        assert float((K - want).abs().max()) <= KERNEL_ABS
