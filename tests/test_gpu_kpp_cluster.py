"""Kernel k-means++ in one launch (mini-batches of a few MB): picks against the
oracle's draws from the same stream.

The device forms D^2 from FP32 kernel values, so a draw whose target lies
within their error of an interval's end may give a neighbour; a pick is
accepted when the oracle's running sum at it is within 1e-5 of the total of the
target (the kernel tolerance summed over the samples), given the picks before
it.  Row lengths for each number of lanes to a row, one group of 32 samples and
one past it, more groups than the cluster has warps, more groups than a chunk of
the pick's scan, all samples equal (every D^2 zero)."""

import numpy as np
import pytest

from oracle import kkm_oracle as O
from synth import blobs

pytestmark = pytest.mark.gpu


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x, np.float32)).to("cuda:0")


@pytest.mark.parametrize("N,d,C", [(32, 3, 5), (33, 8, 20), (1000, 12, 9), (4100, 30, 16), (4097, 60, 7),
                                   (9000, 100, 12), (2500, 300, 6), (700, 1030, 4)])
@pytest.mark.parametrize("kind", ["rbf", "linear"])
def test_picks(lib, N, d, C, kind):
    X, _ = blobs(N, d, 6, workload=61, problem=N + d)
    sigma = 2.0 * np.sqrt(d)
    seed = 5
    got = lib.kkm_debug_kmeanspp(_dev(X), C, seed, kind, sigma)
    kpp, _, _ = O.rng_streams(seed, 1)
    k = O.Kernel(O.KIND_RBF if kind == "rbf" else O.KIND_LINEAR, float(np.float32(sigma)))
    Xo = X.astype(np.float64)
    ks = k.self_terms(Xo)
    assert got[0] == int(np.floor(kpp.u01() * N))
    D2 = np.full(N, np.inf)
    for r in range(1, C):
        m = int(got[r - 1])
        D2 = np.maximum(np.minimum(D2, ks - 2.0 * k(Xo, Xo[m:m + 1])[:, 0] + ks[m]), 0.0)
        prefix = np.cumsum(D2)
        target, slack = kpp.u01() * prefix[-1], 1e-5 * prefix[-1]
        p = int(got[r])
        before = prefix[p - 1] if p else 0.0
        assert before - slack <= target <= prefix[p] + slack, (r, p)
        assert D2[p] > 0.0


def test_equal_samples_take_the_lowest_unchosen(lib):
    X = np.ones((100, 16), np.float32)
    got = lib.kkm_debug_kmeanspp(_dev(X), 6, 3, "rbf", 1.0)
    rest = [i for i in range(100) if i != got[0]][:5]
    assert list(got[1:]) == rest
