"""kkm_assign_noalloc gives the bits of kkm_assign for RBF and linear models, as
the header says, on either kernel block: FFMA (short rows, few references) and
the FP16 slices (more references, longer rows), with the
references in one block of its scratch, in several, and one past a block's end,
and with rows that the slices do not hold among references and samples."""

import numpy as np
import pytest

from synth import mnist_like

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind,n,d,C,mode", [
    ("rbf", 700, 100, 5, "supports"), ("rbf", 1025, 784, 10, "supports"), ("rbf", 3001, 130, 8, "supports"),
    ("rbf", 1300, 66, 6, "supports"), ("rbf", 600, 130, 40, "medoids"), ("rbf", 900, 1024, 33, "medoids"), ("rbf", 500, 48, 5, "supports"),
    ("rbf", 300, 200, 7, "medoids"), ("linear", 800, 90, 5, "supports")])
@pytest.mark.parametrize("wide", [False, True])
def test_same_bits_as_assign(lib, kind, n, d, C, mode, wide):
    import torch
    X, _ = mnist_like(n + 1024, d, 10, problem=n + d)
    if wide:
        g = np.random.default_rng(n)
        for r in np.nonzero(g.random(len(X)) < 0.1)[0]:
            X[r] *= np.float32(0.001)
            X[r, g.integers(0, d)] = 2.0
    S, Q = (torch.from_numpy(np.ascontiguousarray(x, np.float32)).to("cuda:0") for x in (X[:n], X[n:]))
    _, model = lib.kkm_fit(S, C, 1, 1.0, kind, 0.0 if kind == "linear" else 0.3 * np.sqrt(d), iters=2, seed=1)
    for M in (1, 127, 1024):
        q = Q[:M].contiguous()
        lab = torch.empty(M, dtype=torch.int32, device="cuda:0")
        dist = torch.empty(M, dtype=torch.float32, device="cuda:0")
        lib.kkm_assign_noalloc(model, q, lab, dist, mode)
        want_lab, want_dist = lib.kkm_assign(model, q, mode)
        assert torch.equal(lab, want_lab) and torch.equal(dist, want_dist)
