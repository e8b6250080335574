"""The near-tie re-score of the tensor-core loop, whose FP32 kernel values are
kept from iteration to iteration.

Rows of a class that two clusters share are near ties in every iteration, and
their labels (and those of the landmarks among them) keep moving, so the kept
values are read again, extended and read under other cluster lists.  A fit of
t iterations has to give what t separate steps give, each of which starts with
nothing kept: the sums are the same values in the same order, so labels, Omega
and the changed counts agree bit for bit.  Shapes: a ragged last tile, one
landmark word and several blocks of 1,024 landmarks, row lengths whose last
chunk of 32 products is short, rows whose FP32 block values are kept already
(at most 128 values), and the largest C of the loop."""

import numpy as np
import pytest

from synth import mnist_like

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,s,C,d,classes,prec", [
    (1037, 0.5, 8, 136, 3, "bf16"), (2600, 0.8, 12, 260, 4, "bf16"), (130, 0.2, 4, 200, 2, "bf16"),
    (1500, 0.75, 16, 150, 5, "fp8"), (2300, 0.5, 9, 64, 3, "bf16"), (3000, 1.0, 2, 784, 1, "bf16")])
def test_kept_values_equal_fresh_ones(lib, N, s, C, d, classes, prec):
    import torch
    X, _ = mnist_like(N, d, classes, problem=N + d)
    Xd = torch.from_numpy(X).to("cuda:0")
    p = lib.KKM_BF16 if prec == "bf16" else lib.KKM_FP8
    sig = float(np.float32(0.32 * np.sqrt(d)))
    iters, seed = 7, 11
    init = np.arange(C) * (N // C)

    def fit(t):
        return lib.kkm_fit(Xd, C, 1, s, "rbf", sig, iters=t, seed=seed, precision=p, iteration="tc", early_stop=False,
                           init_medoids=init)

    u = fit(0)[0].cpu().numpy()
    _, L = lib.kkm_minibatch_plan(N, 1, s, seed, 0)
    omega, changed = [], []
    for _ in range(iters):
        step = lib.kkm_debug_step(Xd, L, u, C, "rbf", sig, precision=p, iteration="tc")
        u = step["u"]
        omega.append(step["omega"])
        changed.append(step["changed"])
    lab, model = fit(iters)
    om, ch = model.trace()
    assert np.array_equal(ch, changed)
    assert np.array_equal(om, omega)
    assert np.array_equal(lab.cpu().numpy(), u)
    assert sum(changed) > 0 or classes == 1
