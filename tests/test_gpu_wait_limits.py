"""The bounded waits of the tensor-core kernel blocks, run out of polls.

A wait that gives up has to end the whole CTA: every warp leaves its loop, the
copies and MMAs in flight are waited for, tensor memory is freed, the call
returns KKM_ETIMEOUT and the next call gives the values it always gives (a
kernel that kept its tensor memory would hold that call up).  With no polls
every wait gives up at once; with a few, waits run out at places that differ
from CTA to CTA and from run to run, while copies and MMAs are in flight, or
not at all.  Several tiles a CTA and several chunks of a row."""

import numpy as np
import pytest

from synth import md_trajectory, mnist_like

pytestmark = pytest.mark.gpu

ETIMEOUT = 5


def _limits(lib, A, B, kind, sigma, precision, n_atoms=0):
    import torch
    want = lib.kkm_kernel_matrix(A, B, kind, sigma, n_atoms, precision=precision)
    with pytest.raises(lib.KKMError) as e:
        lib.kkm_kernel_matrix(A, B, kind, sigma, n_atoms, precision=precision, polls=0)
    assert e.value.status == ETIMEOUT
    for polls in (1, 2, 5, 20, 100):
        try:
            got = lib.kkm_kernel_matrix(A, B, kind, sigma, n_atoms, precision=precision, polls=polls)
            assert torch.equal(got, want)
        except lib.KKMError as err:
            assert err.status == ETIMEOUT
        assert torch.equal(lib.kkm_kernel_matrix(A, B, kind, sigma, n_atoms, precision=precision), want)


@pytest.mark.parametrize("nA,nB,d", [(600, 20001, 600), (100, 500, 300)])
def test_fp32_slices(lib, nA, nB, d):
    import torch
    X, _ = mnist_like(nA + nB, d, 5, problem=nA + d)
    Xd = torch.from_numpy(np.ascontiguousarray(X, np.float32)).to("cuda:0")
    _limits(lib, Xd[:nA].contiguous(), Xd[nA:].contiguous(), "rbf", 0.3 * np.sqrt(d), lib.KKM_FP32)


@pytest.mark.parametrize("prec", ["bf16", "fp8"])
def test_reduced_precision_block(lib, prec):
    import torch
    X, _ = mnist_like(20601, 600, 5, problem=6)
    Xd = torch.from_numpy(np.ascontiguousarray(X, np.float32)).to("cuda:0")
    _limits(lib, Xd[:600].contiguous(), Xd[600:].contiguous(), "rbf", 7.0, lib.KKM_BF16 if prec == "bf16" else lib.KKM_FP8)


def test_md_screen(lib):
    import torch
    F, _ = md_trajectory(n_frames=9600, n_atoms=70, n_states=5, dwell=50.0, workload=83)
    Xd = torch.from_numpy(np.ascontiguousarray(F.reshape(9600, -1), np.float32)).to("cuda:0")
    _limits(lib, Xd[:600].contiguous(), Xd[600:].contiguous(), "rmsd", 1.5, lib.KKM_FP32, 70)
