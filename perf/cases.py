"""Cases that time this framework as its users run it: trajectory-kNN rarity scores of
gridded daily fields, from a quick look at one year on a coarse grid to 75 years on the
0.25-degree European grid, and the gradient of the scores.

Inputs are SLP-like anomalies built on the GPU from a seed, with the recipe of `synth`:
random low-wavenumber Fourier modes whose coefficients follow an AR(1) process of
persistence 0.8, a standard deviation of 10 hPa.
"""
import math
import random

import numpy as np
import torch

import paper_2603_02059_gb300 as tk

YEAR = 365.25


def listed():
    return [
        # a first look: one year of a coarse grid, where launches and latency count
        dict(name="year_8x8", kind="forward", n=365, h=8, w=8, L=3, k=5, precision="split_bf16"),
        # five years of a 16 x 32 grid: a short record on a global coarse grid
        dict(name="5y_16x32", kind="forward", n=1826, h=16, w=32, L=3, k=10,
             precision="split_bf16"),
        # the 1-degree European grid: 30 years, and the 75 years of the headline workload
        dict(name="30y_1deg", kind="forward", n=10957, h=46, w=81, L=5, k=10,
             precision="split_bf16"),
        dict(name="75y_1deg", kind="forward", n=27394, h=46, w=81, L=5, k=20,
             precision="split_bf16"),
        # the headline workload from page-locked host arrays to host arrays
        dict(name="75y_1deg_host", kind="host", n=27394, h=46, w=81, L=5, k=20,
             precision="split_bf16"),
        # the headline workload in plain FP32, the accuracy reference of a study
        dict(name="75y_1deg_fp32", kind="forward", n=27394, h=46, w=81, L=5, k=20,
             precision="fp32"),
        # the largest: 75 years on the 0.25-degree grid
        dict(name="75y_quarter", kind="forward", n=27394, h=181, w=321, L=5, k=20,
             precision="split_bf16"),
        # fields reduced to a few dozen components
        dict(name="75y_4x8", kind="forward", n=27394, h=4, w=8, L=5, k=20,
             precision="split_bf16"),
        # an odd region and day count, cosine-of-latitude weights, the single-product form
        dict(name="20y_weighted_bf16", kind="forward", n=7301, h=45, w=79, L=7, k=15,
             precision="bf16", weighted=True),
        # several trajectory lengths of one record in one call ("what if L were ...")
        dict(name="30y_lengths", kind="multi", n=10957, h=46, w=81, lengths="3,5,7,10", k=10,
             precision="split_bf16"),
        # an ensemble of uneven records (regions, members) in one call
        dict(name="ensemble", kind="batched", series=12, n=3650, n_hi=14000, h=46, w=81, mix=7,
             precision="split_bf16"),
        # the gradient of the summed scores at fixed neighbours, 30 years
        dict(name="30y_backward", kind="backward", n=10957, h=46, w=81, L=5, k=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost_ms(c):
    """A rough time of a case in ms, to keep drawn cases below the largest listed one."""
    n, d = (c.get("n_hi") or c["n"]), c["h"] * c["w"]
    per = {"fp32": 5e-11, "bf16": 2e-12}.get(c.get("precision"), 2.5e-12)
    one = n * n * (d * per + 3e-9 * (1 + c.get("k", 20) / 20))
    times = c.get("series", 1) * 0.6 if c["kind"] == "batched" else \
        1 + 0.6 * c["lengths"].count(",") if c["kind"] == "multi" else 1
    return one * max(1.0, times)


def draw(rng):
    while True:
        kind = rng.choices(["forward", "host", "multi", "batched", "backward", "train"],
                           [10, 2, 2, 2, 3, 1])[0]
        d = _log(rng, 16, 60000)
        h = max(1, int(round(math.sqrt(d) * rng.uniform(0.4, 1.0))))
        c = dict(kind=kind, n=_log(rng, 300, 27400), h=h, w=max(1, round(d / h)))
        L = rng.choice([1, 2, 3, 3, 4, 5, 5, 5, 6, 7, 8, 10, 10, 12, 17])
        k = rng.choice([1, 5, 5, 8, 10, 10, 15, 20, 20, 20, 30, 40, 64])
        if kind == "backward":
            c |= dict(L=L, k=k)
        else:
            c["precision"] = rng.choices(["split_bf16", "fp32", "bf16"], [7, 2, 1])[0]
        if kind in ("forward", "host", "train"):
            c |= dict(L=L, k=k)
        if kind == "forward" and rng.random() < 0.25:
            c["weighted"] = True
        if kind == "multi":
            c |= dict(lengths=",".join(map(str, sorted(rng.sample(range(1, 13),
                                                                  rng.randint(2, 5))))), k=k)
        if kind == "batched":
            c |= dict(series=rng.randint(2, 20), n_hi=min(27400, int(c["n"] * rng.uniform(1.2, 4))),
                      mix=rng.randrange(1000))
        n = c.get("n_hi") or c["n"]
        held = n * c["h"] * c["w"] * c.get("series", 1)
        if _cost_ms(c) < 75.0 and held < 1.6e9:
            return c


# ------------------------------------------------------------------------ inputs

def _fields(n, h, w, seed):
    """[n, h w] float32 anomalies on the GPU, from the seed alone."""
    rng = np.random.default_rng(seed)
    modes, kmax, phi = 40, 4, 0.8
    ks = rng.integers(-kmax, kmax + 1, size=(4 * modes, 2))
    ks = ks[(ks != 0).any(axis=1)][:modes].astype(np.float64)
    amp = 1.0 / (1.0 + (ks ** 2).sum(axis=1))
    phase = rng.uniform(0.0, 2.0 * np.pi, size=modes)
    eps = rng.standard_normal((n, 2 * modes)) * math.sqrt(0.5)
    c = np.empty_like(eps)
    c[0] = eps[0]
    eps *= math.sqrt(1.0 - phi * phi)
    for t in range(1, n):
        c[t] = phi * c[t - 1] + eps[t]
    dev = torch.device("cuda")
    y, x = torch.meshgrid(torch.arange(h, dtype=torch.float64, device=dev),
                          torch.arange(w, dtype=torch.float64, device=dev), indexing="ij")
    kt = torch.from_numpy(ks).to(dev)
    arg = 2.0 * math.pi * (kt[:, 0, None] * x.reshape(1, -1) / w
                           + kt[:, 1, None] * y.reshape(1, -1) / h)
    arg += torch.from_numpy(phase).to(dev)[:, None]
    a = torch.from_numpy(amp).to(dev)[:, None]
    basis = torch.cat([a * torch.cos(arg), -a * torch.sin(arg)]).float()
    X = torch.from_numpy(c).to(dev).float() @ basis
    # standard deviation 10 (a mode of amplitude a and a unit coefficient has variance a^2 / 2)
    return X.mul_(10.0 / math.sqrt(float((amp ** 2).sum()) / 2.0))


def _weights(h, w):
    lat = torch.linspace(30.0, 75.0, h, device="cuda") * (math.pi / 180.0)
    return torch.cos(lat).float().repeat_interleave(w).contiguous()


def _shapes(case):
    """(n, L, k) of every series of an ensemble: part of the case, not of the seed."""
    rng = random.Random(case["mix"])
    return [(rng.randint(case["n"], case["n_hi"]), rng.randint(2, 10), rng.choice([5, 10, 20]))
            for _ in range(case["series"])]


def _outs(m, k, device, pin=False):
    o = dict(device=device, pin_memory=pin) if pin else dict(device=device)
    return (torch.empty((m, k), dtype=torch.int32, **o), torch.empty((m, k), **o),
            torch.empty((m,), **o))


def _state_fields(case, seed):
    return _fields(case["n"], case["h"], case["w"], seed)


def _neighbours(X, L, k):
    """[M, k] int32 neighbour sets in plain torch (what a backward pass is given)."""
    return _exact_knn(X, [(L, k)], None, torch.float32)[0][0]


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "batched":
        shapes = _shapes(case)
        s["series"] = [(_fields(n, case["h"], case["w"], seed * 64 + b), L, k, L - 1)
                       for b, (n, L, k) in enumerate(shapes)]
        s["outs"] = [_outs(n - L + 1, k, "cuda") for n, L, k in shapes]
        return s
    X = _state_fields(case, seed)
    if kind == "host":
        s["X"] = torch.empty(X.shape, pin_memory=True).copy_(X)
        s["out"] = _outs(case["n"] - case["L"] + 1, case["k"], "cpu", pin=True)
        return s
    s["X"] = X
    if kind == "backward":
        s["idx"] = _neighbours(X, case["L"], case["k"])
        gen = torch.Generator(device="cuda").manual_seed(seed)
        s["g"] = torch.rand(s["idx"].shape[0], device="cuda", generator=gen) + 0.5
    elif kind == "train":
        s["X"].requires_grad_(True)
    elif case.get("weighted"):
        s["handle"] = tk.Handle()
        s["handle"].set_grid_weights(_weights(case["h"], case["w"]))
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "forward":
        return tk.knn_scores(s["X"], c["L"], c["k"], precision=c["precision"],
                             handle=s.get("handle"))
    if kind == "host":
        return tk.knn_scores_host(s["X"], c["L"], c["k"], precision=c["precision"], out=s["out"])
    if kind == "multi":
        return tk.knn_scores_multi(s["X"], [(int(L), c["k"], None) for L in
                                            c["lengths"].split(",")], precision=c["precision"])
    if kind == "batched":
        return tk.knn_scores_batched(s["series"], precision=c["precision"], outs=s["outs"])
    if kind == "backward":
        return tk.score_backward(s["X"], c["L"], c["k"], s["idx"], s["g"])
    X = s["X"]
    X.grad = None
    score = tk.TrakNNScore.apply(X, c["L"], c["k"], None, c["precision"])
    score.sum().backward()
    return score, X.grad


# ------------------------------------------------------------------ work and values

def _settings(case):
    """(n, L, k) of every result set of the case."""
    if case["kind"] == "batched":
        return _shapes(case)
    if case["kind"] == "multi":
        return [(case["n"], int(L), case["k"]) for L in case["lengths"].split(",")]
    return [(case["n"], case["L"], case["k"])]


def work(case):
    """Each input read and each output written once; the Gram matrix of each record's
    days once (its upper triangle); the gradient: each neighbour pair's L day differences."""
    d = case["h"] * case["w"]
    sets = _settings(case)
    records = sets if case["kind"] == "batched" else sets[:1]
    nbytes = sum(4 * n * d for n, _, _ in records)
    lists = sum((n - L + 1) * (8 * k + 4) for n, L, k in sets)
    gram = sum(n * (n + 1) * d for n, _, _ in records)
    if case["kind"] in ("backward", "train"):
        n, L, k = sets[0]
        m = n - L + 1
        grad = 2 * 2 * m * k * L * d
        if case["kind"] == "backward":
            return dict(bytes=2 * nbytes + m * (4 * k + 4), flops=grad)
        return dict(bytes=2 * nbytes + 4 * m, flops=gram + grad)
    return dict(bytes=nbytes + lists, flops=gram)


def _exact_knn(X, settings, weights, dtype=torch.float64):
    """[(idx, dist, score)] of every (L, k), by plain blocks of the distance matrix."""
    X = X.to(dtype)
    X = X - X.mean(dim=0)
    if weights is not None:
        X = X * weights.to(dtype).sqrt()
    n = X.shape[0]
    norm = (X * X).sum(dim=1)
    lmax = max(L for L, _ in settings)
    found = [[] for _ in settings]
    rows = 1024
    for t0 in range(0, n, rows):
        a1 = min(n, t0 + rows + lmax - 1)
        S = torch.addmm(norm[None, :], X[t0:a1], X.T, alpha=-2.0).add_(norm[t0:a1, None])
        for (L, k), out in zip(settings, found):
            m = n - L + 1
            r = min(rows, m - t0)
            if r <= 0:
                continue
            dist = S[:r, :m].clone()
            for i in range(1, L):
                dist += S[i:i + r, i:i + m]
            t = torch.arange(t0, t0 + r, device=X.device)
            j = torch.arange(m, device=X.device)
            dist.masked_fill_((t[:, None] - j[None, :]).abs() < L, math.inf)
            v, i = dist.topk(k, dim=1, largest=False, sorted=True)
            out.append((i.int(), v.clamp_(min=0.0)))
    got = []
    for out in found:
        v = torch.cat([o[1] for o in out])
        got.append((torch.cat([o[0] for o in out]), v, v.mean(dim=1)))
    return got


def _exact_gradient(X, L, k, idx, g):
    X = X.double()
    m, j = idx.shape[0], idx.long()
    dX = torch.zeros_like(X)
    for r in range(k):
        for i in range(L):
            diff = X[i:i + m] - X[j[:, r] + i]
            diff *= (2.0 / k) * g.double()[:, None]
            dX[i:i + m] += diff
            dX.index_add_(0, j[:, r] + i, diff, alpha=-1.0)
    return dX


def exact(case, seed):
    d = case["h"] * case["w"]
    sets = _settings(case)
    records = sets if case["kind"] == "batched" else sets[:1]
    if sum(2 * n * n * d for n, _, _ in records) > 1.2e13:
        return None
    if case["kind"] == "batched":
        got = []
        for b, (n, L, k) in enumerate(sets):
            X = _fields(n, case["h"], case["w"], seed * 64 + b)
            got += [(None, v, s) for _, v, s in _exact_knn(X, [(L, k)], None)]
        return got
    X = _state_fields(case, seed)
    if case["kind"] == "backward":
        n, L, k = sets[0]
        if 4 * n * d * L * k > 4e12:
            return None
        gen = torch.Generator(device="cuda").manual_seed(seed)
        g = torch.rand(n - L + 1, device="cuda", generator=gen) + 0.5
        return _exact_gradient(X, L, k, _neighbours(X, L, k), g)
    w = _weights(case["h"], case["w"]) if case.get("weighted") else None
    got = [(None, v, s) for _, v, s in _exact_knn(X, [(L, k) for _, L, k in sets], w)]
    if case["kind"] == "multi":
        return got
    if case["kind"] == "train":
        return got[0][2], None  # the gradient depends on near ties of the neighbour sets
    out = got[0]
    return tuple(v.cpu() if v is not None else None for v in out) if case["kind"] == "host" \
        else out
