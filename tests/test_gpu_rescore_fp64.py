"""The near-tie re-score of the tensor-core loop against 64-bit values.

The re-score gives f_hat (Eq. 17) of a row's candidate clusters from FP32 kernel
values; g_hat (Eq. 16) is the loop's own, from the stored block.  So here: f_hat
in 64 bits, g_hat as the loop has it.  For rows whose low-precision margin lies well inside the re-score's window, the
label of a fit's next iteration has to be the 64-bit one wherever the 64-bit
margin is clear of FP32 rounding (1e-4 of the second distance, the repository's
rule for labels).  Each shape must show that the re-score ran and mattered: rows
inside the window, rows that stay there while landmarks move between clusters
(so kept values are read again under other lists), and rows whose low-precision
argmin is another cluster than the 64-bit one."""

import numpy as np
import pytest

from synth import mnist_like
from tests.helpers import rel_margin

pytestmark = pytest.mark.gpu


def _two_least(d):
    p = np.partition(d, 1, axis=1)
    return p[:, 0], p[:, 1]


@pytest.mark.parametrize("N,s,C,d,classes,prec,tau", [
    (2600, 0.8, 12, 260, 4, "bf16", 1e-3), (1037, 0.5, 8, 136, 3, "bf16", 1e-3), (1500, 0.75, 16, 150, 5, "fp8", 3e-2)])
def test_flagged_rows_get_the_64_bit_label(lib, N, s, C, d, classes, prec, tau):
    import torch
    X, _ = mnist_like(N, d, classes, problem=N + d)
    Xd = torch.from_numpy(X).to("cuda:0")
    p = lib.KKM_BF16 if prec == "bf16" else lib.KKM_FP8
    sig = float(np.float32(0.32 * np.sqrt(d)))
    seed, init = 11, np.arange(C) * (N // C)
    _, L = lib.kkm_minibatch_plan(N, 1, s, seed, 0)
    x = X.astype(np.float64)
    n2 = (x * x).sum(1)
    K = np.exp(-np.maximum(n2[:, None] + n2[None, L] - 2 * x @ x[L].T, 0) / (2 * sig * sig))
    K[L, np.arange(len(L))] = 1.0

    def fit(t):
        lab, _ = lib.kkm_fit(Xd, C, 1, s, "rbf", sig, iters=t, seed=seed, precision=p, iteration="tc", early_stop=False,
                             init_medoids=init)
        return lab.cpu().numpy()

    u, before, stayed, moved, overruled = fit(0), None, 0, 0, 0
    for t in range(1, 7):
        step = lib.kkm_debug_step(Xd, L, u, C, "rbf", sig, precision=p, iteration="tc")
        low = 1.0 - 2.0 * step["fhat"].astype(np.float64) + step["ghat"]
        low[:, step["n"] == 0] = np.inf
        best, second = _two_least(low)
        inside = second - best < 0.5 * tau * np.maximum(np.abs(second), 1.0)
        Z = (u[L][:, None] == np.arange(C)).astype(np.float64)
        nj = Z.sum(0)
        with np.errstate(invalid="ignore"):
            d64 = np.where(nj > 0, 1.0 - 2.0 * (K @ Z / nj) + step["ghat"], np.inf)
        check = inside & (rel_margin(d64) > 1e-4)
        new = fit(t)
        assert np.array_equal(new[check], d64.argmin(1)[check])
        overruled += int((check & (low.argmin(1) != d64.argmin(1))).sum())
        if before is not None:
            stayed += int((inside & before).sum())
        moved += int((new[L] != u[L]).sum())
        before, u = inside, new
    assert stayed > 0 and moved > 0 and overruled > 0, (stayed, moved, overruled)
