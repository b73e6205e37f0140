"""Workloads that measure this library through its public entry points.

Each case is a plain dict; ``prepare`` makes its inputs and the handles a
program keeps between calls (index, codebooks, network weights), ``run`` makes
one pass through ``paper_2404_00774_gb300.binding``, ``work`` counts the bytes
and operations the pass cannot do without, and ``exact`` computes the same
results in 64 bits with plain torch.  Sizes are those of the synthetic
workloads (``synth.WORKLOADS``) and of the benchmark's studies, or generic.
"""
from __future__ import annotations

import math

import torch

DEV = "cuda"
LAMBDA = 1.0        # weight of the SOAR penalty (Theorem 3.1); one spill everywhere
SPILLS = 1


# ------------------------------------------------------------------ the cases

def listed():
    glove = dict(kind="search", mix="anisotropic", n=1_183_514, d=100, c=2000, dtype="f32", score="full", k=10, t=14)
    return [
        # the smallest index with a small batch: every launch and allocation shows
        dict(glove, name="tiny_search", mix="isotropic", n=20_000, d=64, c=64, nq=100, t=4),
        # one interactive query against a million-point index: latency
        dict(glove, name="online_search", nq=1),
        # the headline batch: 10 000 queries, top 10 at recall 0.9
        dict(glove, name="glove_search", nq=10_000),
        # a ten times larger index stored in bf16 (ten thousand partitions)
        dict(glove, name="bf16_search", mix="isotropic", n=10_000_000, d=96, c=10_000, dtype="bf16", nq=10_000, t=5),
        # one batch as the serving loop forms it: top 100, every request with its own probe count
        # (the serving workload's shape with a tenth of its points and partitions)
        dict(glove, name="serving_batch", mix="isotropic", n=10_000_000, d=128, c=4000, dtype="bf16", nq=1024, k=100,
             t=512, t_lo=32),
        # the FP8 layout: codes of every copy scored, the best 1 000 rescored exactly
        dict(glove, name="fp8_search", mix="isotropic", n=10_000_000, d=96, c=10_000, dtype="bf16", score="fp8",
             nq=10_000, t=6, rescore=1000),
        # the 4-bit PQ layout: table look-ups over every copy's code, the best 100 rescored exactly
        dict(glove, name="pq4_search", score="pq4", nq=10_000, rescore=100),
        # two-level selection over many small partitions
        dict(glove, name="multilevel_search", mix="isotropic", n=3_000_000, d=96, c=30_000, dtype="bf16", nq=10_000,
             t=5, c2=550, t1=4),
        # the probe count of every query predicted by the network inside the search
        dict(glove, name="learned_search", nq=10_000, t=32, hidden=256),
        # one training step of that network (top-64 features), bf16 products as the training loop uses them
        dict(kind="train_step", name="probe_train_step", batch=4096, d_in=164, hidden=256, bf16=True),
        # the whole build of a million-point index: codebook, spilled assignment, inverted lists
        dict(kind="build", name="index_build", mix="anisotropic", n=1_183_514, d=100, c=2000, dtype="f32", iters=10),
        # exact ground truth of a query batch by brute force
        dict(kind="brute", name="ground_truth", mix="anisotropic", n=1_183_514, d=100, dtype="f32", nq=10_000, k=10),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    what = rng.choice(["full", "full", "full", "wide", "fp8", "pq4", "multilevel", "learned", "train_step", "build",
                       "brute"])
    if what == "train_step":
        return dict(kind=what, batch=log(500, 8192), d_in=rng.randint(70, 200), hidden=rng.choice([64, 128, 200, 256]),
                    bf16=rng.random() < 0.75)
    c = log(40, 2500)
    per = rng.randint(300, 900)                              # points per partition
    n, d = c * per + rng.randint(0, 99), rng.randint(48, 128)
    dtype, mix = rng.choice(["f32", "f32", "bf16"]), rng.choice(["isotropic", "anisotropic"])
    if what == "build":
        return dict(kind=what, mix=mix, n=min(n, 1_200_000), d=min(d, 104), c=c, dtype=dtype, iters=rng.randint(2, 8))
    if what == "brute":
        return dict(kind=what, mix=mix, n=min(n, 1_200_000), d=d, dtype=dtype, nq=log(16, 8000),
                    k=rng.choice([1, 10, 10, 32, 100]))
    case = dict(kind="search", mix=mix, n=n, d=d, c=c, dtype=dtype, score="full", nq=log(1, 10_000),
                k=rng.choice([1, 5, 10, 10, 16]), t=min(c, log(2, 32)))
    if what == "wide":                                       # serving batches: large k, per-query probe counts
        case.update(nq=log(16, 1024), k=rng.choice([20, 50, 100]), t=min(c, log(40, 400)))
        case.update(t_lo=max(1, case["t"] // 16))
    elif what in ("fp8", "pq4"):
        case.update(score=what, d=d - d % 2, k=10, rescore=rng.choice([50, 100, 333, 1000]))
    elif what == "multilevel":
        c = log(2000, 20_000)
        case.update(c=c, n=c * rng.randint(60, 120), c2=max(16, c // 60), t=rng.randint(3, 12), t1=rng.randint(2, 8),
                    k=10)
    elif what == "learned":
        case.update(t=min(c, 32), hidden=rng.choice([128, 256]), k=10)
    return case


# ------------------------------------------------------------------ inputs

def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _mixture(mix, rows, d, comps, g):
    """Unit vectors of a Gaussian mixture of equally likely components: broad anisotropic ones whose spectra span
    two decades (the shape of word vectors), or tight isotropic ones (sigma 0.3)."""
    comps = max(16, min(comps, rows // 100))
    each = -(-rows // comps)
    order = torch.randperm(comps * each, generator=g, device=DEV)[:rows]
    v = torch.randn((comps, each, d), generator=g, device=DEV)
    if mix == "anisotropic":
        eig = torch.exp(math.log(0.01) * torch.rand((comps, 1, d), generator=g, device=DEV))
        turn = torch.randn((comps, d, d), generator=g, device=DEV) / math.sqrt(d)
        v = torch.bmm(v * eig.sqrt(), turn) + 0.2 * torch.randn((comps, 1, d), generator=g, device=DEV)
    else:
        v = torch.randn((comps, 1, d), generator=g, device=DEV) + 0.3 * v
    v = v.reshape(-1, d)[order]
    return v / v.norm(dim=1, keepdim=True)


def _points(case, seed):
    """(X, Q): datapoints in the stored type and fp32 queries, drawn from one mixture."""
    g = _generator(seed)
    nq = case.get("nq", 0)
    # 4 (broad) or 10 (tight) partitions to a component, as in the library's synthetic workloads
    comps = case.get("c", 2000) // (4 if case["mix"] == "anisotropic" else 10)
    v = _mixture(case["mix"], case["n"] + nq, case["d"], comps, g)
    X = v[nq:].to(torch.bfloat16 if case["dtype"] == "bf16" else torch.float32)
    return X.contiguous(), v[:nq].clone(), g


def _blocks(n, width, most=1 << 28):
    step = max(1, most // max(1, width))
    return [(i, min(n, i + step)) for i in range(0, n, step)]


def _nearest(X, C):
    """Nearest centroid of every row."""
    half = 0.5 * (C * C).sum(1)
    out = torch.empty(X.shape[0], dtype=torch.int64, device=DEV)
    for i, j in _blocks(X.shape[0], C.shape[0]):
        out[i:j] = (X[i:j].to(C.dtype) @ C.T - half).argmax(1)
    return out


def _lloyd(X, C, iters, dtype):
    """Lloyd steps; means in 64 bits, an empty cluster keeps its centroid."""
    for _ in range(iters):
        a = _nearest(X, C.to(dtype))
        cnt = torch.bincount(a, minlength=C.shape[0])[:, None]
        s = torch.zeros(C.shape, dtype=torch.float64, device=DEV).index_add_(0, a, X.double())
        C = torch.where(cnt > 0, s / cnt.clamp(min=1), C.double())
    return C


def _codebook(X, c, g):
    """A codebook trained on a sample, as a program that already has one would load it.  Entries are rounded to
    a grid of 2^-12, so that the order of the additions does not show."""
    S = X[: min(X.shape[0], max(20 * c, 10_000))].float()
    C = _lloyd(S, S[torch.randperm(S.shape[0], generator=g, device=DEV)[:c]], 3, torch.float32)
    return (torch.round(C * 4096) / 4096).float()


def _pq_codebooks(X, C, g):
    """PQ centres [d/2][16][2] of the residuals of a sample (three Lloyd steps per subspace, on a grid of 2^-12)."""
    S = X[:20_000].float()
    r = (S - C[_nearest(S, C)]).view(S.shape[0], -1, 2).transpose(0, 1).contiguous()      # [m][rows][2]
    B = r[:, torch.randperm(r.shape[1], generator=g, device=DEV)[:16]]
    for _ in range(3):
        hit = torch.nn.functional.one_hot(torch.cdist(r, B).argmin(2), 16).double()       # [m][rows][16]
        cnt = hit.sum(1)[:, :, None]
        B = torch.where(cnt > 0, hit.transpose(1, 2) @ r.double() / cnt.clamp(min=1), B.double()).float()
        B = torch.round(B * 4096) / 4096
    return B.contiguous()


def _network(d_in, hidden, g):
    """Weights of a probe-count network (W1 | b1 | W2 | b2 | W3 | b3) whose outputs spread around log 8."""
    def u(rows, cols):
        return (2 * torch.rand((rows, cols), generator=g, device=DEV) - 1) * math.sqrt(6.0 / cols)

    def bias(m):
        return 0.1 * torch.randn((m,), generator=g, device=DEV)

    return torch.cat([u(hidden, d_in).reshape(-1), bias(hidden), u(hidden, hidden).reshape(-1), bias(hidden),
                      0.5 * u(1, hidden).reshape(-1), torch.full((1,), math.log(8.0), device=DEV)])


def _inputs(case, seed):
    """What a case's pass starts from, the same for ``prepare`` and ``exact``."""
    if case["kind"] == "train_step":
        g = _generator(seed)
        B, d_in = case["batch"], case["d_in"]
        q = torch.nn.functional.normalize(torch.randn((B, d_in - 64), generator=g, device=DEV), dim=1)
        s = (0.3 + 0.5 * torch.rand((B, 64), generator=g, device=DEV)).sort(1, descending=True)[0]
        target = torch.log(1.0 + torch.floor(20 * torch.rand((B,), generator=g, device=DEV) ** 2))
        return dict(Z=torch.cat([q, s], 1).contiguous(), target=target, params=_network(d_in, case["hidden"], g))
    X, Q, g = _points(case, seed)
    if case["kind"] == "build":
        init = torch.randperm(case["n"], generator=g, device=DEV)[: case["c"]].sort()[0].int()
        return dict(X=X, init=init)
    if case["kind"] == "brute":
        return dict(X=X, Q=Q)
    C = _codebook(X, case["c"], g)
    s = dict(X=X, Q=Q, C=C)
    if case["score"] == "pq4":
        s["B"] = _pq_codebooks(X, C, g)
    if case.get("t_lo"):
        s["tpq"] = torch.randint(case["t_lo"], case["t"] + 1, (case["nq"],), generator=g, device=DEV).int()
    if case.get("c2"):
        s["init2"] = torch.randperm(case["c"], generator=g, device=DEV)[: case["c2"]].sort()[0].int()
    if case.get("hidden"):
        s["params"] = _network(case["d"] + case["t"], case["hidden"], g)
    return s


# ------------------------------------------------------------------ the measured calls

def prepare(case, seed):
    from paper_2404_00774_gb300 import binding as soar
    s = _inputs(case, seed)
    s["case"] = case
    if case["kind"] == "train_step":
        s["grads"], s["m1"], s["m2"] = (torch.zeros_like(s["params"]) for _ in range(3))
        s["loss"], s["step"] = torch.zeros((1,), device=DEV), 0
    if case["kind"] == "search":
        X, C = s.pop("X"), s["C"]
        A = soar.soar_assign(X, C, LAMBDA, SPILLS)
        if case["score"] == "pq4":
            s["index"] = soar.soar_index_build_pq(X, C, A, s["B"])
        else:
            mode = soar.SOAR_SCORE_FP8 if case["score"] == "fp8" else soar.SOAR_SCORE_F32
            s["index"] = soar.soar_index_build(X, C, A, mode)
        if case.get("c2"):
            s["coarse"] = soar.soar_index_build_coarse(s["index"], case["c2"], 4, s["init2"], LAMBDA, SPILLS)
    return s


def run(state):
    from paper_2404_00774_gb300 import binding as soar
    case = state["case"]
    if case["kind"] == "train_step":
        d_in, hidden = case["d_in"], case["hidden"]
        state["step"] += 1
        soar.soar_mlp_backward(state["params"], d_in, hidden, state["Z"], state["target"], case["bf16"],
                               state["grads"], state["loss"])
        soar.soar_mlp_adam(state["params"], state["grads"], state["m1"], state["m2"], state["step"], 1e-3)
        return dict(grads=state["grads"], loss=state["loss"])
    if case["kind"] == "build":
        C = soar.soar_train_centroids(state["X"], case["c"], case["iters"], state["init"])
        A = soar.soar_assign(state["X"], C, LAMBDA, SPILLS)
        ix = soar.soar_index_build(state["X"], C, A)
        out = dict(centroids=C, assign=A, offsets=ix.offsets(), ids=ix.ids(), vectors=ix.vectors())
        ix.close()
        return out
    if case["kind"] == "brute":
        ids, scores = soar.soar_exact_mips(state["X"], state["Q"], case["k"])
        return dict(ids=ids, scores=scores)
    ix, Q, k, t = state["index"], state["Q"], case["k"], case["t"]
    if case.get("c2"):
        ids, scores = soar.soar_search_multilevel(ix, state["coarse"], Q, k, t, case["t1"])
    elif case.get("hidden"):
        ids, scores, counts = soar.soar_search_learned(ix, Q, k, t, state["params"], case["hidden"], 1.0, t)
        return dict(ids=ids, scores=scores, counts=counts)
    else:
        ids, scores = soar.soar_search(ix, Q, k, t, state.get("tpq"), case.get("rescore", 0))
    return dict(ids=ids, scores=scores)


def work(case):
    """Bytes: inputs and outputs once; a search reads the partitions its batch touches once (never more than the
    index) and the codebook.  Operations: the dot products of the probed rows, the selection's scores, the
    assignments' scores."""
    if case["kind"] == "train_step":
        D, H, B = case["d_in"], case["hidden"], case["batch"]
        p = H * D + H + H * H + H + H + 1
        return dict(bytes=4.0 * (B * (D + 1) + 8 * p), flops=6.0 * B * (H * D + H * H + H) - 2.0 * B * H * D)
    n, d = case["n"], case["d"]
    es = 4 if case["dtype"] == "f32" else 2
    if case["kind"] == "build":
        c, it = case["c"], case["iters"]
        return dict(bytes=float(n * d * es * (it + 2) + 2 * n * (d * es + 8) + 8 * c * d),
                    flops=2.0 * n * c * d * (it + 3))
    nq, k = case["nq"], case["k"]
    if case["kind"] == "brute":
        return dict(bytes=float(n * d * es + nq * (4 * d + 12 * k)), flops=2.0 * n * nq * d)
    c, per = case["c"], (1 + SPILLS) * n / case["c"]
    t = (case["t"] + case["t_lo"]) / 2 if case.get("t_lo") else 0.4 * case["t"] if case.get("hidden") else case["t"]
    row = {"full": d * es, "fp8": d + 4, "pq4": d // 4}[case["score"]] + 4
    touched = c * (1 - (1 - t / c) ** nq)                     # distinct partitions the batch touches
    scored = case["t1"] * 2 * c / case["c2"] + case["c2"] if case.get("c2") else c
    by = touched * per * row + 4 * d * min(c, scored * nq) + nq * (4 * d + 12 * k)
    fl = 2.0 * nq * d * (scored + t * per)
    if case.get("rescore"):
        by += min(n, nq * case["rescore"]) * d * es
        fl += 2.0 * nq * d * case["rescore"]
    return dict(bytes=float(by), flops=float(fl))


# ------------------------------------------------------------------ the same in 64 bits

def _spilled(X, C):
    """[n][2]: the nearest centroid and the SOAR spill (64 bits where that is quick, else 32)."""
    T = torch.float64 if X.shape[0] * C.shape[0] < 1 << 33 else torch.float32
    C = C.to(T)
    first = _nearest(X, C)
    out = torch.stack([first, first], 1)
    for i, j in _blocks(X.shape[0], 2 * C.shape[0]):
        x, f = X[i:j].to(T), first[i:j]
        r = x - C[f]
        r /= r.norm(dim=1, keepdim=True).clamp(min=1e-30)
        loss = (C * C).sum(1) - 2 * x @ C.T + LAMBDA * ((x * r).sum(1, keepdim=True) - r @ C.T) ** 2
        out[i:j, 1] = loss.scatter_(1, f[:, None], float("inf")).argmin(1)
    return out


def _e4m3(V):
    """(code values, scales) of every row."""
    scale = V.abs().amax(1, keepdim=True) / 448
    scale = torch.where(scale > 0, scale, torch.ones_like(scale))
    return (V / scale).to(torch.float8_e4m3fn).float(), scale


def _best_of_union(case, Q, X, A, probes, approx):
    """Scores of the best k of every query's probed union: the best R by approx(q0, q1, order), then 64 bits.
    `order` [rows][c]: the place of every partition in the query's probe order (large: not probed)."""
    nq, k, n, c = Q.shape[0], case["k"], X.shape[0], case["c"]
    R = min(n, case.get("rescore", k + 22))
    out = torch.full((nq, k), float("-inf"), dtype=torch.float64, device=DEV)
    for i, j in _blocks(nq, n):
        order = torch.full((j - i, c + 1), 30_000, dtype=torch.int16, device=DEV)
        place = torch.arange(probes.shape[1], device=DEV, dtype=torch.int16).expand(j - i, -1).contiguous()
        order.scatter_(1, probes[i:j] % (c + 1), place)       # -1 (not probed) falls into the last column
        order = order[:, :c]
        s, idx = approx(i, j, order).topk(R, dim=1)
        exact = torch.einsum("qd,qrd->qr", Q[i:j].double(), X[idx].double())
        exact = exact.masked_fill(torch.isinf(s), float("-inf"))
        out[i:j, : min(k, R)] = exact.topk(min(k, R), dim=1)[0]
    return out


def exact(case, seed):
    if case["kind"] == "search" and case["n"] * case["nq"] > 3e10 * (1 if case.get("rescore", 0) > 200 else 6):
        return None
    s = _inputs(case, seed)
    if case["kind"] == "train_step":
        return _exact_train_step(case, s)
    X = s["X"]
    if case["kind"] == "build":
        if case["n"] * case["c"] * case["d"] * case["iters"] > 4e12:
            return None
        C = _lloyd(X, X[s["init"].long()].double(), case["iters"], torch.float64)
        return dict(centroids=C, assign=None, offsets=None, ids=None, vectors=None)
    Q, n = s["Q"], case["n"]
    Xf = X.float()
    if case["kind"] == "brute":
        A = torch.zeros((n, 1), dtype=torch.int64, device=DEV)
        probes = torch.zeros((case["nq"], 1), dtype=torch.int64, device=DEV)
        scores = _best_of_union(dict(case, c=1), Q, Xf, A, probes, lambda i, j, order: Q[i:j] @ Xf.T)
        return dict(ids=None, scores=scores)
    C, t = s["C"], case["t"]
    A = _spilled(X, C)
    S = Q.double() @ C.double().T
    if case["score"] == "fp8":
        (q8, qs), (c8, cs), (x8, xs) = _e4m3(Q), _e4m3(C), _e4m3(Xf)
        S = (q8.double() @ c8.double().T) * qs * cs.T
    if case.get("c2"):
        C2 = _lloyd(C, C[s["init2"].long()].double(), 4, torch.float64).float()
        A2 = _spilled(C, C2)
        first = (Q.double() @ C2.double().T).topk(case["t1"], dim=1)[1]
        seen = torch.zeros((case["nq"], case["c2"]), dtype=torch.bool, device=DEV).scatter_(1, first, True)
        S = S.masked_fill(~(seen[:, A2[:, 0]] | seen[:, A2[:, 1]]), float("-inf"))
    ranked, probes = S.topk(t, dim=1)
    probes = probes.masked_fill(torch.isinf(ranked), -1)
    counts = s.get("tpq")
    if case.get("hidden"):
        Z = torch.cat([Q, ranked.float()], 1)
        y = _forward(s["params"], Z, case["hidden"], True)[-1]
        counts = torch.exp(y).ceil().clamp(1, t)
    if counts is not None:
        probes = probes.masked_fill(torch.arange(t, device=DEV) >= counts[:, None], -1)

    def approx(i, j, order):
        o0, o1 = order[:, A[:, 0]], order[:, A[:, 1]]
        if case["score"] == "fp8":
            v = (q8[i:j] @ x8.T) * xs.T
        elif case["score"] == "pq4":
            v = torch.where(o0 <= o1, Q[i:j] @ rows[0].T, Q[i:j] @ rows[1].T)
        else:
            v = Q[i:j] @ Xf.T
        return v.masked_fill(torch.minimum(o0, o1) >= 30_000, float("-inf"))

    rows = []
    if case["score"] == "pq4":                                # every copy as its codes spell it
        for col in range(2):
            base = C[A[:, col]]
            r = (Xf - base).view(n, -1, 2)
            parts = []
            for m in range(r.shape[1]):
                B = s["B"][m]
                d0, d1 = r[:, m, :1] - B[:, 0], r[:, m, 1:] - B[:, 1]
                parts.append(B[(d0 * d0 + d1 * d1).argmin(1)])
            rows.append(base + torch.cat(parts, 1))
    out = dict(ids=None, scores=_best_of_union(case, Q, Xf, A, probes, approx))
    if case.get("hidden"):
        out["counts"] = None
    return out


def _forward(params, Z, H, bf16):
    """Pre-activations and activations of the network in 64 bits; with bf16 every product's operands are rounded."""
    D = Z.shape[1]

    def r(v):
        return v.float().to(torch.bfloat16).double() if bf16 else v.double()

    W1, b1, W2, b2, W3, b3 = torch.split(params, [H * D, H, H * H, H, H, 1])
    h1 = torch.relu(r(Z) @ r(W1).view(H, D).T + b1.double())
    h2 = torch.relu(r(h1) @ r(W2).view(H, H).T + b2.double())
    return h1, h2, r(h2) @ r(W3) + b3.double()


def _exact_train_step(case, s):
    Z, target, H, B = s["Z"], s["target"].double(), case["hidden"], case["batch"]
    D = case["d_in"]

    def r(v):
        return v.float().to(torch.bfloat16).double() if case["bf16"] else v.double()

    _, _, W2, _, W3, _ = torch.split(s["params"], [H * D, H, H * H, H, H, 1])
    h1, h2, y = _forward(s["params"], Z, H, case["bf16"])
    gy = 2 * (y - target) / B
    ga2 = r(gy)[:, None] * r(W3)[None, :] * (h2 > 0)
    ga1 = (r(ga2) @ r(W2).view(H, H)) * (h1 > 0)
    grads = [r(ga1).T @ r(Z), ga1.sum(0), r(ga2).T @ r(h1), ga2.sum(0), r(h2).T @ r(gy), gy.sum()[None]]
    return dict(grads=torch.cat([v.reshape(-1) for v in grads]), loss=((y - target) ** 2).mean()[None])
