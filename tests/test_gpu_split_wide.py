"""Rows that the slices of the FP32 Gaussian block do not hold: NaN and Inf, a
squared norm outside the FP32 range, a largest value far above the rest.  Their
pairs come from the FFMA sums, everyone else's from the tensor cores, so a value
depends on its two rows alone.

Tolerance against 64 bits per entry: the norms and the dot product are FP32
roundings of sums of size |a|^2 + |b|^2 (at most 4 + 4 units of 2^-24 of it), so
K is off by at most 8 * 2^-24 (|a|^2 + |b|^2) / (2 sigma^2) plus the
exponential's own 2^-21."""

import numpy as np
import pytest

from synth import mnist_like

pytestmark = pytest.mark.gpu


def _dev(x):
    import torch
    return torch.from_numpy(np.ascontiguousarray(x, np.float32)).to("cuda:0")


def _matrix(lib, A, B, sigma):
    return lib.kkm_kernel_matrix(_dev(A), _dev(B), "rbf", sigma).cpu().numpy()


def _check(K, A, B, sigma):
    a, b = A.astype(np.float64), B.astype(np.float64)
    norms = (a * a).sum(1)[:, None] + (b * b).sum(1)[None, :]
    s2 = 2 * float(np.float32(sigma)) ** 2
    off = np.abs(K - np.exp(-np.maximum(norms - 2 * a @ b.T, 0) / s2))
    assert np.all(off <= 2.0 ** -21 + 8 * 2.0 ** -24 * norms / s2)


def _widen(X, which, g):
    """A value 2,000 times the others in the rows `which` (scaled back, so that
    one bandwidth suits every row)."""
    X = X.copy()
    for r in which:
        X[r] *= np.float32(0.001)
        X[r, g.integers(0, X.shape[1])] = 2.0
    return X


@pytest.mark.parametrize("nA,nB,d", [(33, 1, 128), (1025, 127, 66), (300, 700, 131), (257, 4100, 784), (513, 300, 100)])
@pytest.mark.parametrize("share", ["one", "few", "half", "most", "all"])
def test_wide_rows_against_64_bits(lib, nA, nB, d, share):
    g = np.random.default_rng(nA + d)
    X, _ = mnist_like(nA + nB, d, 5, problem=nA + d)
    pick = {"one": lambda n: [n - 1], "few": lambda n: np.nonzero(g.random(n) < 0.03)[0],
            "half": lambda n: np.nonzero(g.random(n) < 0.5)[0], "most": lambda n: np.nonzero(g.random(n) < 0.97)[0],
            "all": lambda n: np.arange(n)}[share]
    A, B = _widen(X[:nA], pick(nA), g), _widen(X[nA:], pick(nB), g)
    sigma = 0.3 * np.sqrt(d)
    _check(_matrix(lib, A, B, sigma), A, B, sigma)
    _check(_matrix(lib, A, X[nA:], sigma), A, X[nA:], sigma)
    _check(_matrix(lib, X[:nA], B, sigma), X[:nA], B, sigma)


def test_a_value_depends_on_its_two_rows_alone(lib):
    g = np.random.default_rng(9)
    X, _ = mnist_like(1700, 200, 5, problem=9)
    A, B, sigma = X[:500], X[500:], 4.0
    K = _matrix(lib, A, B, sigma)
    A2, B2 = _widen(A, [3, 400], g), _widen(B, [0, 700], g)
    B2[17, 3] = np.nan
    B2[40, 0] = np.inf
    A2[250, 199] = -np.inf
    K2 = _matrix(lib, A2, B2, sigma)
    ra, rb = np.setdiff1d(np.arange(500), [3, 400, 250]), np.setdiff1d(np.arange(1200), [0, 700, 17, 40])
    assert np.array_equal(K2[np.ix_(ra, rb)], K[np.ix_(ra, rb)])
    # the wide rows' values do not depend on the company either
    sub = _matrix(lib, A2[[3, 400] + list(range(40, 180))], B2[[700, 0]], sigma)
    assert np.array_equal(sub[:2], K2[np.ix_([3, 400], [700, 0])])
    # nor, bit for bit, on how many of them there are (few go 16 to a tile, many 128; 64 is the line)
    for many in (61, 62, 300):
        A4, B4 = _widen(A2, range(4, 4 + many), g), _widen(B2, range(100, 100 + 2 * many), g)
        B4[900:1000] = B2[900:1000]
        K4 = _matrix(lib, A4, B4, sigma)
        keep = [0, 700] + list(range(900, 1000))
        assert np.array_equal(K4[np.ix_([3, 400], keep)], K2[np.ix_([3, 400], keep)])
        clean = np.setdiff1d(np.arange(350, 500), [400])
        assert np.array_equal(K4[np.ix_(clean, [0, 700])], K2[np.ix_(clean, [0, 700])])
    # nor on where the rows lie: unaligned rows of an odd pitch
    import torch
    flat = torch.zeros(1 + A2.size, device="cuda:0")
    flat[1:] = _dev(A2).reshape(-1)
    K3 = lib.kkm_kernel_matrix(flat[1:].view(500, 200), _dev(B2), "rbf", sigma).cpu().numpy()
    assert np.array_equal(K3, K2)


def test_rows_beyond_the_range_of_the_norm(lib):
    """A row whose |x|^2 underflows is at the origin; one whose |x|^2 overflows
    (its norm has no FP32 value) leaves the other rows' values alone."""
    X, _ = mnist_like(400, 96, 4, problem=2)
    A, B = X[:150].copy(), X[150:].copy()
    want = _matrix(lib, A, B, 3.0)
    B[7] *= np.float32(1e33)
    B[9] *= np.float32(1e-30)
    K = _matrix(lib, A, B, 3.0)
    keep = np.setdiff1d(np.arange(250), [7])
    _check(K[:, keep], A, B[keep], 3.0)
    assert np.array_equal(np.delete(K, [7, 9], 1), np.delete(want, [7, 9], 1))


@pytest.mark.parametrize("mode,C", [("supports", 6), ("medoids", 40)])
def test_assign_of_wide_rows(lib, mode, C):
    """Wide rows among the references and the samples: each sample's result is
    that of a call of its own, and the distances are those of kkm_cost's FFMA
    block to FP32 rounding."""
    g = np.random.default_rng(3)
    X, _ = mnist_like(3700, 150, 10, problem=3)
    X = _widen(X, np.nonzero(g.random(3700) < 0.1)[0], g)
    S, Q = _dev(X[:700]), _dev(X[700:])
    _, model = lib.kkm_fit(S, C, 1, 1.0, "rbf", 3.0, iters=2, seed=1)
    lab, dist = lib.kkm_assign(model, Q, mode)
    for rows in ([5], list(range(130)), list(range(1000, 2300))):
        la, da = lib.kkm_assign(model, Q[rows].contiguous(), mode)
        assert np.array_equal(la.cpu().numpy(), lab[rows].cpu().numpy())
        assert np.array_equal(da.cpu().numpy(), dist[rows].cpu().numpy())
    cost = lib.kkm_cost(model, Q, mode)
    entry = 2.0 ** -21 + 8 * 2.0 ** -24 * 2 * float((X * X).sum(1).max()) / 18.0  # of a kernel value, as above
    assert abs(cost - float(dist.double().sum())) <= 3000 * 2 * entry


def test_assign_in_several_chunks(lib):
    """More rows than one chunk of kernel values holds (22,369 to 6,000 supports): the
    references' slices and lists are those of the first chunk, the wide samples
    each chunk's own."""
    g = np.random.default_rng(4)
    X, _ = mnist_like(6000 + 50000, 130, 10, problem=4)
    X = _widen(X, np.nonzero(g.random(len(X)) < 0.02)[0], g)
    S, Q = _dev(X[:6000]), _dev(X[6000:])
    _, model = lib.kkm_fit(S, 5, 1, 1.0, "rbf", 3.0, iters=1, seed=1)
    lab, dist = lib.kkm_assign(model, Q)
    lab, dist = lab.cpu().numpy(), dist.cpu().numpy()
    for a, b in ((0, 20000), (20000, 40000), (40000, 50000), (22360, 22380)):
        la, da = lib.kkm_assign(model, Q[a:b].contiguous())
        assert np.array_equal(la.cpu().numpy(), lab[a:b]) and np.array_equal(da.cpu().numpy(), dist[a:b])
