"""Admission of assign jobs whose block comes from FP16 slices: a budget that
leaves room for the job with the FP32 rows of the FFMA block (the estimate such
jobs always had) admits it; the slices are then made in parts, and labels and
distances are kkm_assign's, bit for bit."""

import numpy as np
import pytest

from synth import mnist_like

pytestmark = pytest.mark.gpu

SLACK, UNIT, STRIP = 8 << 20, 64, 512


def _ffma_estimate(M, d, dp, nL, C):
    ldm = -(-M // 32) * 32
    units = -(-nL // UNIT) + C
    return (4 * M * d + 8 * M + 4 * ldm * (dp + 1) + 4 * nL * ldm + 4 * units * ldm + 8 * units * -(-ldm // STRIP)
            + SLACK)


@pytest.mark.parametrize("M,n,d", [(5, 3000, 784), (700, 1100, 203)])
def test_tight_budget_admits_and_gives_the_same_bits(lib, M, n, d):
    import torch
    C = 6
    X, _ = mnist_like(n + M, d, C, problem=d)
    X[n + 2, :] *= np.float32(0.001)
    X[n + 2, 7] = 2.0  # a row that the slices do not hold
    S, Q = (torch.from_numpy(np.ascontiguousarray(x, np.float32)).to("cuda:0") for x in (X[:n], X[n:]))

    def model():
        return lib.kkm_fit(S, C, 1, 1.0, "rbf", 0.3 * np.sqrt(d), iters=2, seed=1)[1]

    srv = lib.Server(budget_bytes=1 << 33, n_workers=1)
    srv.add_model(model())
    resident = srv.stats()["bytes_in_use"]
    srv.close()
    want_lab, want_dist = lib.kkm_assign(model(), Q)
    torch.cuda.synchronize()
    srv = lib.Server(budget_bytes=resident + _ffma_estimate(M, d, -(-d // 8) * 8, n, C), n_workers=1)
    mid = srv.add_model(model())
    t = srv.submit_assign(mid, Q)
    assert srv.stats()["refused"] == 0
    status, out, _, err = srv.wait(t)
    assert status == 0, err
    lab, dist = out
    assert np.array_equal(np.asarray(torch.as_tensor(lab).cpu()), want_lab.cpu().numpy())
    assert np.array_equal(np.asarray(torch.as_tensor(dist).cpu()), want_dist.cpu().numpy())
    assert srv.stats()["peak_bytes"] <= resident + _ffma_estimate(M, d, -(-d // 8) * 8, n, C)
    srv.close()
