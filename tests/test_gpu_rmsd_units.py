"""The MD kernel block (tensor-core screen, then the exact residual of the near
pairs) against the oracle at the edges of its tiles: 40 samples x 80 references
of the screen, 16 x 16 pairs of the exact pass, ten samples to a lane quarter,
eight atoms to a stage and 64 atoms to a K step; no pair near, every pair near,
and references in an order unlike the samples'.  Tolerance: the kernel
tolerance of the parity tests (1e-5 absolute); pairs whose true value is below
the screen's threshold may be exactly 0."""

import numpy as np
import pytest

from oracle import kkm_oracle as O
from synth import md_trajectory
from tests.helpers import KERNEL_ABS

pytestmark = pytest.mark.gpu


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x, np.float32)).to("cuda:0")


@pytest.mark.parametrize("nA,nB,atoms,states,dwell", [
    (32, 1, 8, 2, 5.0), (33, 41, 9, 3, 4.0), (80, 40, 64, 4, 7.0), (81, 39, 65, 3, 9.0), (79, 121, 23, 8, 3.0),
    (161, 257, 30, 5, 11.0), (96, 160, 12, 2, 1e9)])
@pytest.mark.parametrize("sigma", [0.5, 1.5])
def test_block_against_oracle(lib, nA, nB, atoms, states, dwell, sigma):
    F, _ = md_trajectory(nA + nB, atoms, n_states=states, dwell=dwell, workload=77, problem=nA + nB)
    g = np.random.default_rng(nA)
    pick = g.permutation(nA + nB)
    A, B = F[pick[:nA]], F[np.sort(pick[nA:])]
    k = O.Kernel(O.KIND_RMSD, sigma, atoms)
    want = k(A.reshape(nA, -1).astype(np.float64), B.reshape(nB, -1).astype(np.float64))
    got = lib.kkm_kernel_matrix(_dev(A.reshape(nA, -1)), _dev(B.reshape(nB, -1)), "rmsd", sigma, atoms).cpu().numpy()
    off = np.abs(got - want)
    assert np.max(off) <= KERNEL_ABS, float(np.max(off))
    assert np.all(want[got == 0.0] <= KERNEL_ABS)
    one_state = dwell > 1e6
    if not one_state and sigma == 0.5:
        assert np.any(got == 0.0)
    if one_state and sigma == 1.5:
        assert np.all(got > 0.0)


def test_values_do_not_depend_on_the_other_pairs(lib):
    """A pair's value is the same bits in any block that holds it."""
    F, _ = md_trajectory(500, 40, n_states=4, dwell=20.0, workload=78, problem=1)
    A, B = _dev(F[:200].reshape(200, -1)), _dev(F[200:].reshape(300, -1))
    K = lib.kkm_kernel_matrix(A, B, "rmsd", 1.5, 40).cpu().numpy()
    a, b = np.arange(3, 199, 4), np.arange(5, 300, 7)
    part = lib.kkm_kernel_matrix(A[a].contiguous(), B[b].contiguous(), "rmsd", 1.5, 40).cpu().numpy()
    assert np.array_equal(part, K[np.ix_(a, b)])
