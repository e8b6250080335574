"""Calls that fit in device memory without the scratch that makes them faster:
kernel blocks beside the scratch of the FFMA block and not beside that of the
FP16 slices (half as much again), and reduced-precision fits without the re-score's
kept values.  They run, in parts or without, with the same bits.

Device memory is filled until the free part lies between the two (inputs and
outputs are there already); no call is made that has to fail.  In a process of
its own, whose memory pool is trimmed before each call, so that what is free is
what the call gets."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = """
import ctypes
import torch
from paper_1710_03013_gb300 import kkm

kkm.load()
rt = ctypes.CDLL("libcudart.so.13")


def trim():
    pool = ctypes.c_void_p()
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    assert rt.cudaMemPoolTrimTo(pool, ctypes.c_size_t(0)) == 0
    torch.cuda.empty_cache()


def squeezed(call, free):
    torch.cuda.synchronize()
    trim()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - free, dtype=torch.uint8, device="cuda")
    out = call()
    del fill
    trim()
    return out


g = torch.Generator(device="cuda")
g.manual_seed(4)
GB = 1 << 30
# matrix: rows 6,000 + 150,000 of 2,048 values; FFMA rows 1.19 GiB, slices 1.79, the output beside them
A = torch.rand(6000, 2048, generator=g, device="cuda")
B = torch.rand(150000, 2048, generator=g, device="cuda")
B[77, 5] = 3e4
A[5000, 9] = float("nan")
out = torch.empty(6000, 150000, device="cuda")


def matrix():
    k = kkm._kernel("rbf", 9.0, 0)
    kkm._check(kkm.load().kkm_kernel_matrix(A.data_ptr(), 6000, B.data_ptr(), 150000, 2048, ctypes.byref(k), 0,
                                            out.data_ptr(), None))


squeezed(matrix, int(1.5 * GB))
tight = out.clone()
matrix()
assert torch.equal(out, tight)
del out, tight, B
# assign: one chunk of 40,000 rows of 16,384 values to 3,000 supports; FFMA rows 2.44 GiB, slices 3.94, block 0.45
S = torch.rand(3000, 16384, generator=g, device="cuda")
_, model = kkm.kkm_fit(S, 3, 1, 1.0, "rbf", 30.0, iters=0, seed=1, init_medoids=range(3))
Q = torch.rand(40000, 16384, generator=g, device="cuda")
Q[123, 45] = 1e3
res = []
lab = [torch.empty(40000, dtype=torch.int32, device="cuda") for _ in range(2)]
dist = [torch.empty(40000, device="cuda") for _ in range(2)]


def assign(i):
    kkm._check(kkm.load().kkm_assign(model.handle, Q.data_ptr(), 40000, kkm.MODE["supports"], lab[i].data_ptr(),
                                     dist[i].data_ptr(), None))


assign(1)
for free in (3.5, 4.1, 4.3, 4.42):  # the last ones hold the slices, but not the block beside them
    squeezed(lambda: assign(0), int(free * GB))
    assert torch.equal(lab[0], lab[1]) and torch.equal(dist[0], dist[1])
    lab[0].zero_()
print("both ran in parts")
"""


def test_calls_that_fit_beside_the_ffma_scratch_run(lib):
    done = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, done.stderr[-2000:]
    assert "both ran in parts" in done.stdout


FIT = """
import ctypes
import numpy as np
import torch
from paper_1710_03013_gb300 import kkm
from synth import mnist_like

kkm.load()
rt = ctypes.CDLL("libcudart.so.13")
pool = ctypes.c_void_p()
assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
RESERVED, RESERVED_HIGH = 5, 6


def trim():
    torch.cuda.synchronize()
    assert rt.cudaMemPoolTrimTo(pool, ctypes.c_size_t(0)) == 0
    torch.cuda.empty_cache()


for d, classes, C in ((200, 5, 12), (100, 4, 9)):
    X, _ = mnist_like(18000, d, classes, problem=d)
    X = torch.from_numpy(np.ascontiguousarray(X, np.float32)).to("cuda")

    def fit():
        lab, model = kkm.kkm_fit(X, C, 1, 0.16, "rbf", 0.32 * d ** 0.5, iters=6, seed=3, precision=kkm.KKM_BF16,
                                 iteration="tc", early_stop=False)
        return (lab.cpu().numpy(),) + tuple(model.trace())

    fit()
    trim()
    zero = ctypes.c_uint64(0)
    assert rt.cudaMemPoolSetAttribute(pool, RESERVED_HIGH, ctypes.byref(zero)) == 0
    want = fit()
    high = ctypes.c_uint64(0)
    assert rt.cudaMemPoolGetAttribute(pool, RESERVED_HIGH, ctypes.byref(high)) == 0
    trim()
    kept = 18000 * 2880 * 4  # the values alone
    for short in (kept // 2, kept // 4, 32 << 20, 8 << 20, 2 << 20):  # to a little less than all of it
        free = high.value - short
        fill = torch.empty(torch.cuda.mem_get_info()[0] - free, dtype=torch.uint8, device="cuda")
        got = fit()
        again = ctypes.c_uint64(0)
        assert rt.cudaMemPoolGetAttribute(pool, RESERVED, ctypes.byref(again)) == 0
        assert again.value <= free
        del fill
        trim()
        assert want[2][1:].sum() > 0
        for a, b in zip(got, want):
            assert np.array_equal(a, b)
print("both fits ran without kept values")
"""


def test_fits_run_without_the_kept_values(lib):
    done = subprocess.run([sys.executable, "-c", FIT], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert done.returncode == 0, done.stderr[-2000:]
    assert "ran without kept values" in done.stdout
