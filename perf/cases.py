"""Performance cases: what a program does with this library, through its public entry points.

Five kinds of call, each over the sizes at which the library is used:

  fit      kkm_fit of one data set (feature vectors, blobs or MD frames), device-resident input, labels, model and trace read back;
  batch    kkm_fit_batch of many small, uneven problems;
  assign   kkm_assign of new samples to a fitted model (its landmark supports or its medoids);
  matrix   kkm_kernel_matrix, the kernel block as a call of its own.

`listed()` names the sizes that stand for each kind, `draw()` spreads over the same ranges.  Data follow the library's
workloads: clipped class templates quantised to k/255 (feature vectors), Gaussian blobs, and Markov-jump trajectories of
random-coil conformations in random poses (MD frames).
"""

import math

import numpy as np
import torch

from paper_1710_03013_gb300 import kkm

DEV = "cuda"
PRECISION = {"fp32": kkm.KKM_FP32, "bf16": kkm.KKM_BF16, "fp8": kkm.KKM_FP8}


def listed():
    return [
        # The headline fit: MNIST-shaped features on the reduced-precision path, every iteration run, every class found
        # (a refit from known medoids, one of each class).
        dict(name="fit_features_bf16", kind="fit", data="features", N=60000, d=784, C=10, B=4, s=0.2, iters=30,
             precision="bf16", sampling="stride", early_stop=False, sigma=0.0, init=True),
        # The same with k-means++ and more clusters than classes, as in a search for C: classes are split, and the rows
        # between two halves are near ties.
        dict(name="fit_features_bf16_split", kind="fit", data="features", N=60000, d=784, C=12, B=4, s=0.2, iters=30,
             precision="bf16", sampling="stride", early_stop=False, sigma=0.0),
        # The same fit at the default precision.
        dict(name="fit_features_fp32", kind="fit", data="features", N=60000, d=784, C=10, B=4, s=0.2, iters=30,
             precision="fp32", sampling="stride", early_stop=False, sigma=0.0),
        # The MD workload: half a million 300-atom frames, RMSD kernel.
        dict(name="fit_frames", kind="fit", data="frames", N=500000, d=900, C=8, B=20, s=0.05, iters=25,
             precision="fp32", sampling="stride", early_stop=False, sigma=1.5),
        # The smallest fit in use: exact kernel k-means (every sample a landmark), launches and host work count.
        dict(name="fit_blobs_small", kind="fit", data="blobs", N=2000, d=16, C=5, B=1, s=1.0, iters=20,
             precision="fp32", sampling="stride", early_stop=True, sigma=4.0),
        # A quarter of the batched workload: many uneven problems side by side.
        dict(name="batch_64", kind="batch", problems=64, shapes=3, iters=30, precision="bf16"),
        # Serving, the largest request against the largest model: 10,000 frames, 10,000 supports.
        dict(name="assign_frames", kind="assign", data="frames", M=10000, n=10000, d=900, C=8, mode="supports",
             sigma=1.5),
        # Serving, a handful of frames against the smallest model: latency.
        dict(name="assign_frames_few", kind="assign", data="frames", M=32, n=1000, d=900, C=8, mode="supports",
             sigma=1.5),
        # Labelling a held-out set of feature vectors against a model of one mini-batch's landmarks.
        dict(name="assign_features", kind="assign", data="features", M=50000, n=3000, d=784, C=10, mode="supports",
             sigma=9.0),
        # One to a few new samples: the smallest call of all.
        dict(name="assign_features_few", kind="assign", data="features", M=5, n=3000, d=784, C=10, mode="supports",
             sigma=9.0),
        # One mini-batch's kernel block at the default precision, ragged in both directions.
        dict(name="matrix_rbf_fp32", kind="matrix", data="features", nA=3001, nB=15013, d=784, kernel="rbf",
             precision="fp32", sigma=9.0),
        # The tensor-core block of the headline fit.
        dict(name="matrix_rbf_bf16", kind="matrix", data="features", nA=3000, nB=15000, d=784, kernel="rbf",
             precision="bf16", sigma=9.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fit_features", "fit_frames", "fit_blobs", "batch", "assign_frames", "assign_features",
                       "matrix", "matrix"])
    if kind == "fit_features":
        return dict(kind="fit", data="features", N=_log_int(rng, 4000, 60000), d=_log_int(rng, 129, 784),
                    C=rng.randint(5, 20), B=rng.randint(1, 4), s=rng.choice([0.1, 0.2, 0.3]), iters=rng.randint(10, 30),
                    precision=rng.choice(["fp32", "bf16", "fp8"]), sampling=rng.choice(["stride", "block"]),
                    early_stop=rng.random() < 0.5, sigma=0.0)
    if kind == "fit_frames":
        return dict(kind="fit", data="frames", N=_log_int(rng, 5000, 200000), d=3 * _log_int(rng, 22, 300),
                    C=rng.randint(4, 12), B=rng.randint(2, 20), s=rng.choice([0.05, 0.1]), iters=rng.randint(10, 25),
                    precision="fp32", sampling=rng.choice(["stride", "block"]), early_stop=rng.random() < 0.5,
                    sigma=1.5)
    if kind == "fit_blobs":
        return dict(kind="fit", data="blobs", N=_log_int(rng, 1000, 50000), d=rng.randint(8, 128),
                    C=rng.randint(2, 64), B=rng.randint(1, 5), s=rng.choice([0.1, 0.5]), iters=rng.randint(10, 30),
                    precision=rng.choice(["fp32", "bf16"]), sampling="stride", early_stop=rng.random() < 0.5, sigma=0.0)
    if kind == "batch":
        return dict(kind="batch", problems=rng.randint(8, 64), shapes=rng.randint(100, 10**6), iters=rng.randint(10, 30),
                    precision=rng.choice(["fp32", "bf16"]))
    if kind == "assign_frames":
        return dict(kind="assign", data="frames", M=_log_int(rng, 1, 10000), n=_log_int(rng, 1000, 10000),
                    d=3 * _log_int(rng, 22, 300), C=rng.randint(4, 16), mode="supports", sigma=1.5)
    if kind == "assign_features":
        d = _log_int(rng, 16, 1024)
        return dict(kind="assign", data="features", M=_log_int(rng, 1, 50000), n=_log_int(rng, 200, 6000), d=d,
                    C=rng.randint(2, 20), mode=rng.choice(["supports", "supports", "medoids"]),
                    sigma=9.0 * math.sqrt(d / 784))
    kernel = rng.choice(["rbf", "rbf", "linear", "rmsd"])
    if kernel == "rmsd":
        return dict(kind="matrix", data="frames", nA=_log_int(rng, 40, 2000), nB=_log_int(rng, 500, 20000),
                    d=3 * _log_int(rng, 22, 300), kernel="rmsd", precision="fp32", sigma=1.5)
    d = _log_int(rng, 16, 1024)
    return dict(kind="matrix", data="features" if kernel == "rbf" else "blobs", nA=_log_int(rng, 40, 5000),
                nB=_log_int(rng, 500, 20000), d=d, kernel=kernel, precision=rng.choice(["fp32", "fp32", "bf16"]),
                sigma=9.0 * math.sqrt(d / 784))


# ------------------------------------------------------------------ inputs
def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * (seed + 1))
    return g


def _features(g, N, d, classes, templates=None):
    """Class templates (a fifth of the coordinates, values 0.3 to 1) plus noise, clipped to [0, 1], multiples of 1/255."""
    if templates is None:
        mask = torch.rand(classes, d, generator=g, device=DEV) < 0.2
        templates = torch.where(mask, 0.3 + 0.7 * torch.rand(classes, d, generator=g, device=DEV),
                                torch.zeros((), device=DEV))
    y = torch.randint(0, classes, (N,), generator=g, device=DEV)
    y[:min(N, classes)] = torch.arange(min(N, classes), device=DEV)
    X = templates[y] + 0.1 * torch.randn(N, d, generator=g, device=DEV)
    X = torch.round(X.clamp_(0.0, 1.0) * 255.0) / 255.0
    return X, templates


def _blobs(g, N, d, blobs):
    centres = 10.0 * torch.rand(blobs, d, generator=g, device=DEV) - 5.0
    y = torch.randint(0, blobs, (N,), generator=g, device=DEV)
    return centres[y] + torch.randn(N, d, generator=g, device=DEV)


def _frames(g, N, d, states, dwell, refs=None):
    """Trajectory of jumps among random coils (3.8 A bonds), 0.5 A noise, a random rotation and shift for every frame."""
    n = d // 3
    if refs is None:
        step = torch.randn(states, n, 3, generator=g, device=DEV)
        refs = torch.cumsum(3.8 * step / step.norm(dim=2, keepdim=True), dim=1)
        refs = refs - refs.mean(dim=1, keepdim=True)
    jump = torch.rand(N, generator=g, device=DEV) < 1.0 / dwell
    jump[:states] = True
    visit = torch.cumsum(jump.to(torch.int64), 0) - 1
    state = torch.randint(0, states, (N,), generator=g, device=DEV)
    state[:states] = torch.arange(states, device=DEV)
    state = state[visit]
    X = torch.empty(N, n, 3, device=DEV)
    for a in range(0, N, 65536):
        b = min(N, a + 65536)
        q = torch.randn(b - a, 4, generator=g, device=DEV)
        w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
        R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                         2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                         2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
        f = refs[state[a:b]] + 0.5 * torch.randn(b - a, n, 3, generator=g, device=DEV)
        X[a:b] = torch.bmm(f, R.transpose(1, 2)) + 20.0 * torch.rand(b - a, 1, 3, generator=g, device=DEV) - 10.0
    return X.view(N, d), refs


def _batch_shapes(case):
    """Shapes of the batched workload: N log-uniform in 1e3..5e4, d in 8, 32, 64, 128, C in 2..64, B = ceil(N / 1e4)."""
    r = np.random.Generator(np.random.PCG64(case["shapes"]))
    out = []
    for _ in range(case["problems"]):
        N = int(round(math.exp(r.uniform(math.log(1e3), math.log(5e4)))))
        out.append(dict(N=N, d=int(r.choice([8, 32, 64, 128])), C=int(r.integers(2, 65)), B=-(-N // 10000),
                        s=float(r.choice([0.1, 0.5]))))
    return out


def _data(case, g, N):
    if case["data"] == "features":
        return _features(g, N, case["d"], 10)[0]
    if case["data"] == "blobs":
        return _blobs(g, N, case["d"], case.get("C", 16))
    return _frames(g, N, case["d"], 8, 2000.0)[0]


def _assign_inputs(case, seed):
    """Rows of the model (its first C rows one of each class, the medoids) and the new samples."""
    g = _generator(seed)
    if case["data"] == "features":
        S, t = _features(g, case["n"], case["d"], case["C"])
        X, _ = _features(g, case["M"], case["d"], case["C"], t)
    else:
        S, refs = _frames(g, case["n"], case["d"], case["C"], 20.0)
        X, _ = _frames(g, max(case["M"], case["C"]), case["d"], case["C"], 50.0, refs)
        X = X[:case["M"]].contiguous()
    return S, X


def prepare(case, seed):
    kind = case["kind"]
    if kind == "fit":
        return {"case": case, "X": _data(case, _generator(seed), case["N"]), "seed": seed}
    if kind == "batch":
        g = _generator(seed)
        problems = []
        for i, p in enumerate(_batch_shapes(case)):
            problems.append(dict(X=_blobs(g, p["N"], p["d"], p["C"]), C=p["C"], B=p["B"], s=p["s"], kind="rbf", sigma=0.0,
                                 iters=case["iters"], seed=seed + i, precision=PRECISION[case["precision"]],
                                 early_stop=False))
        return {"case": case, "problems": problems}
    if kind == "assign":
        S, X = _assign_inputs(case, seed)
        atoms = case["d"] // 3 if case["data"] == "frames" else 0
        # every row a support, labelled by the nearest of one row of each class: the model a program keeps resident
        _, model = kkm.kkm_fit(S, case["C"], 1, 1.0, "rmsd" if atoms else "rbf", case["sigma"], atoms, iters=0, seed=seed,
                               init_medoids=np.arange(case["C"]), labels=False)
        return {"case": case, "X": X, "model": model}
    g = _generator(seed)
    X = _data(case, g, case["nA"] + case["nB"])
    A = torch.zeros(X.shape[0], dtype=torch.bool, device=DEV)  # references spread over the rows, as landmarks are
    A[torch.randperm(X.shape[0], generator=g, device=DEV)[:case["nA"]]] = True
    return {"case": case, "A": X[A], "B": X[~A]}


# ------------------------------------------------------------------ one pass
def _fit_outputs(labels, model, iterations):
    """What a fit gives: labels, medoids (indices, counts, rows), final supports and the trace (zeros after an early stop)."""
    idx, counts, rows = model.medoids()
    sup, ghat, n = model.supports()
    omega, changed = (np.concatenate([t, np.zeros(iterations - len(t), t.dtype)]) for t in model.trace())
    return {"labels": labels, "medoids": idx, "counts": counts, "medoid_rows": rows, "support_labels": sup, "ghat": ghat,
            "support_counts": n, "omega": omega, "changed": changed}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "fit":
        atoms = case["d"] // 3 if case["data"] == "frames" else 0
        labels, model = kkm.kkm_fit(state["X"], case["C"], case["B"], case["s"], "rmsd" if atoms else "rbf", case["sigma"],
                                    atoms, iters=case["iters"], seed=state["seed"], precision=PRECISION[case["precision"]],
                                    sampling=case["sampling"], early_stop=case["early_stop"],
                                    init_medoids=np.arange(case["C"]) if case.get("init") else None)
        return _fit_outputs(labels, model, case["B"] * case["iters"])
    if kind == "batch":
        done = kkm.kkm_fit_batch(state["problems"])
        outs = [_fit_outputs(labels, model, p["B"] * p["iters"]) for p, (labels, model, _) in zip(state["problems"], done)]
        whole = {k: np.concatenate([o[k].reshape(-1) for o in outs]) for k in outs[0] if k != "labels"}
        whole["labels"] = torch.cat([o["labels"] for o in outs])
        return whole
    if kind == "assign":
        labels, dist = kkm.kkm_assign(state["model"], state["X"], mode=case["mode"])
        return {"labels": labels, "dist": dist}
    atoms = case["d"] // 3 if case["kernel"] == "rmsd" else 0
    return kkm.kkm_kernel_matrix(state["A"], state["B"], case["kernel"], case["sigma"], atoms,
                                 precision=PRECISION[case["precision"]])


# ------------------------------------------------------------------ what a pass cannot do without
def _fit_work(N, d, C, B, s, iters, pair):
    Ni = N / B
    L = max(1.0, s * Ni)
    evals = B * (Ni * L + 2 * Ni * C) + (C - 1) * Ni
    return {"bytes": 4.0 * N * d + 4.0 * N, "flops": evals * pair + iters * B * Ni * L}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        each = [_fit_work(p["N"], p["d"], p["C"], p["B"], p["s"], case["iters"], 2.0 * p["d"]) for p in _batch_shapes(case)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    # a pair: 2 d for a dot product; 6 d = 18 per atom for the 3 x 3 correlation of an RMSD
    frames = case["data"] == "frames"
    pair = (6.0 if frames else 2.0) * case["d"]
    if kind == "fit":
        return _fit_work(case["N"], case["d"], case["C"], case["B"], case["s"],
                         1 if case["early_stop"] else case["iters"], pair)
    if kind == "assign":
        n = case["n"] if case["mode"] == "supports" else case["C"]
        return {"bytes": 4.0 * (case["M"] + n) * case["d"] + 8.0 * case["M"], "flops": case["M"] * n * (pair + 1.0)}
    return {"bytes": 4.0 * (case["nA"] + case["nB"]) * case["d"] + 4.0 * case["nA"] * case["nB"],
            "flops": case["nA"] * case["nB"] * pair}


# ------------------------------------------------------------------ 64-bit values
def _sq_euclid(A, B):
    return ((A * A).sum(1)[:, None] + (B * B).sum(1)[None, :] - 2.0 * (A @ B.T)).clamp_(min=0.0)


def _sq_rmsd(A, B):
    """Squared minimum RMSD of all pairs of frames: the largest root of the quaternion matrix's characteristic polynomial
    (Theobald 2005), by Newton's method from above, in 64 bits."""
    n = A.shape[1] // 3
    A = A.view(-1, n, 3)
    B = B.view(-1, n, 3)
    A = A - A.mean(1, keepdim=True)
    B = B - B.mean(1, keepdim=True)
    g = 0.5 * ((A * A).sum((1, 2))[:, None] + (B * B).sum((1, 2))[None, :])
    H = (A.transpose(1, 2).reshape(-1, n) @ B.transpose(1, 2).reshape(-1, n).T).view(len(A), 3, len(B), 3)
    xx, xy, xz, yx, yy, yz, zx, zy, zz = (H[:, i, :, j] / g for i in range(3) for j in range(3))
    c2 = -2.0 * (xx * xx + xy * xy + xz * xz + yx * yx + yy * yy + yz * yz + zx * zx + zy * zy + zz * zz)
    c1 = -8.0 * (xx * (yy * zz - yz * zy) - xy * (yx * zz - yz * zx) + xz * (yx * zy - yy * zx))
    m = [[xx + yy + zz, yz - zy, zx - xz, xy - yx], [yz - zy, xx - yy - zz, xy + yx, zx + xz],
         [zx - xz, xy + yx, yy - xx - zz, yz + zy], [xy - yx, zx + xz, yz + zy, zz - xx - yy]]

    def two(r, i, j):
        return m[r][i] * m[r + 1][j] - m[r][j] * m[r + 1][i]

    c0 = (two(0, 0, 1) * two(2, 2, 3) - two(0, 0, 2) * two(2, 1, 3) + two(0, 0, 3) * two(2, 1, 2)
          + two(0, 1, 2) * two(2, 0, 3) - two(0, 1, 3) * two(2, 0, 2) + two(0, 2, 3) * two(2, 0, 1))
    lam = torch.ones_like(g)
    for _ in range(40):
        p = ((lam * lam + c2) * lam + c1) * lam + c0
        dp = (4.0 * lam * lam + 2.0 * c2) * lam + c1
        lam = lam - torch.where(dp != 0, p / dp, torch.zeros_like(p))
    return (2.0 * g * (1.0 - lam) / n).clamp_(min=0.0)


def _kernel64(A, B, frames, sigma):
    """The Gaussian kernel of all pairs, a few rows of A at a time."""
    A, B = A.double(), B.double()
    rows = max(1, (1 << 22) // max(1, B.shape[0])) if frames else max(1, (1 << 26) // max(1, B.shape[0]))
    sq = _sq_rmsd if frames else _sq_euclid
    return torch.cat([torch.exp(sq(A[a:a + rows], B) / (-2.0 * sigma * sigma)) for a in range(0, A.shape[0], rows)])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("fit", "batch"):
        return None  # tens of seconds to minutes of plain torch: every kernel value, draw and iteration of a whole fit
    sigma = float(case["sigma"])
    if kind == "matrix":
        s = prepare(case, seed)
        if case["kernel"] == "linear":
            return s["A"].double() @ s["B"].double().T
        return _kernel64(s["A"], s["B"], case["kernel"] == "rmsd", sigma)
    S, X = _assign_inputs(case, seed)
    frames, C = case["data"] == "frames", case["C"]
    own = _kernel64(S, S[:C], frames, sigma).argmax(1)
    Z = torch.zeros(case["n"], C, dtype=torch.float64, device=DEV)
    Z[torch.arange(case["n"], device=DEV), own] = 1.0
    n = Z.sum(0)
    KS = _kernel64(S, S, frames, sigma)
    KS.fill_diagonal_(1.0)
    if case["mode"] == "medoids":  # the sample nearest to each support centroid (Eq. 10)
        med = (KS @ Z / n).argmax(0)
        return {"labels": None, "dist": (2.0 - 2.0 * _kernel64(X, S[med], frames, sigma)).min(1).values}
    ghat = ((KS @ Z) * Z).sum(0) / (n * n)
    f = _kernel64(X, S, frames, sigma) @ Z / n
    return {"labels": None, "dist": (1.0 + ghat - 2.0 * f).min(1).values}
