"""Measured cases of the Spectral-LSH compression pass.

Each case is one call of the package's public entry points on inputs made on
the GPU from a seed: the layers of the pass one by one (feature map, Lanczos
and Ritz vectors, SimHash, clusters and macro-tokens) and the pass as a whole
for each backend a program uses (one prompt, token windows, the adaptive
router).  Sizes are those of this repository's workloads (prompts of 512 to
131072 tokens, embedding widths 64 to 5120, 256 to 2048 features, 16 to 64
Lanczos steps), with the preserved last 12 tokens taken off where a layer sees
only the compressible ones; draw() spreads over the same ranges, ragged sizes
among them.

exact() restates each layer in float64 (plain torch and numpy) on the same
inputs.  The pass as a whole has no float64 counterpart where a spectral
backend runs: the sign bits of float32 features and Ritz vectors decide the
clusters, and a clustering from other roundings is another clustering.
"""
import heapq
import math

import numpy as np
import torch

import paper_2607_19368_gb300 as sls

DEV = "cuda"

# tokens, widths: (N, d); the largest stands for a 128k-token prompt
LAST = 12  # trailing tokens a prompt keeps uncompressed by default


def listed():
    return [
        # the reference configuration: a short float32 prompt, where launches
        # and per-step latency count
        {"name": "pass short prompt f32", "kind": "pass", "backend": "global", "B": 1,
         "N": 512, "d": 64, "dtype": "f32", "D": 256, "r": 16, "bits": 8, "rho": 4.0},
        # an 8k prompt of a 7B model through the whole pass
        {"name": "pass 8k prompt", "kind": "pass", "backend": "global", "B": 1,
         "N": 8192, "d": 4096, "dtype": "bf16", "D": 1024, "r": 32, "bits": 12, "rho": 8.0},
        # local windows of 16 tokens, from token ids (the embedding lookup included)
        {"name": "pass 32k local windows", "kind": "tokens", "backend": "local", "B": 1,
         "N": 32768, "d": 3584, "dtype": "bf16", "D": 256, "r": 16, "bits": 0, "rho": 8.0,
         "window": 16, "V": 32768},
        # a batch of prompts through the adaptive router, every window of low
        # redundancy (the chunk path): bound by reading the embeddings
        {"name": "pass adaptive batch", "kind": "pass", "backend": "adaptive", "B": 16,
         "N": 16384, "d": 4096, "dtype": "bf16", "D": 1024, "r": 32, "bits": 0, "rho": 8.0,
         "window": 2048},
        # features of a 32k prompt (bf16 embeddings: the usual type)
        {"name": "features 32k bf16", "kind": "features", "N": 32768 - LAST, "d": 3584,
         "D": 2048, "dtype": "bf16"},
        # float32 embeddings (a program that keeps its embedding table in float32)
        {"name": "features 4k f32", "kind": "features", "N": 4096 - LAST, "d": 2048,
         "D": 1024, "dtype": "f32"},
        # Lanczos and Ritz vectors of an 8k prompt, of a 32k prompt, and of the
        # 2048-token windows of a batch
        {"name": "lanczos 8k", "kind": "lanczos", "N": 8192 - LAST, "d": 4096, "D": 1024,
         "r": 32, "phi": "f32"},
        {"name": "lanczos 32k", "kind": "lanczos", "N": 32768 - LAST, "d": 3584, "D": 2048,
         "r": 64, "phi": "f32"},
        {"name": "lanczos windows", "kind": "windows", "B": 8, "N": 16384 - LAST, "d": 4096,
         "D": 1024, "r": 32, "window": 2048},
        # SimHash of a 128k prompt's Ritz vectors
        {"name": "simhash 128k", "kind": "simhash", "N": 131072 - LAST, "k": 64, "bits": 16},
        # clusters and macro-tokens of a 32k and of an 8k prompt
        {"name": "aggregate 32k", "kind": "aggregate", "N": 32768 - LAST, "d": 3584,
         "dtype": "bf16", "bits": 16, "rho": 16.0, "scheme": "max"},
        {"name": "aggregate 8k", "kind": "aggregate", "N": 8192 - LAST, "d": 4096,
         "dtype": "bf16", "bits": 12, "rho": 8.0, "scheme": "max"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _width(rng, lo, hi, step):
    return max(lo, min(hi, _log(rng, lo, hi) // step * step))


def draw(rng):
    kind = rng.choice(["pass", "tokens", "adaptive", "features", "features", "lanczos", "lanczos",
                       "windows", "simhash", "aggregate", "aggregate"])
    if kind == "pass":  # one prompt; float32 at the reference configuration's widths
        f32 = rng.random() < 0.4
        return {"kind": "pass", "backend": "global", "B": 1, "N": _log(rng, 300, 8192),
                "d": _width(rng, 64, 128 if f32 else 4096, 8), "dtype": "f32" if f32 else "bf16",
                "D": 256 if f32 else rng.choice([256, 512, 1024]), "r": rng.choice([16, 24, 32]),
                "bits": rng.choice([8, 10, 12]), "rho": rng.choice([4.0, 8.0])}
    if kind == "tokens":  # local windows from token ids
        return {"kind": "tokens", "backend": "local", "B": 1, "N": _log(rng, 500, 32768),
                "d": _width(rng, 256, 3584, 8), "dtype": "bf16", "D": 256,
                "r": 16, "bits": 0, "rho": rng.choice([2.0, 4.0, 8.0, 16.0]), "window": 16,
                "V": 32768}
    if kind == "adaptive":
        return {"kind": "pass", "backend": "adaptive", "B": _log(rng, 1, 16),
                "N": _log(rng, 2100, 16384), "d": _width(rng, 1024, 4096, 8), "dtype": "bf16",
                "D": 1024, "r": 32, "bits": 0, "rho": rng.choice([2.0, 4.0, 8.0]), "window": 2048}
    if kind == "features":
        # float32 or bf16 embeddings; any feature count that is a multiple of 4
        f32 = rng.random() < 0.4
        D = rng.choice([256, 512, 1024, 2048]) if rng.random() < 0.6 else _width(rng, 64, 2048, 4)
        return {"kind": "features", "N": _log(rng, 100, 8192 if f32 else 65536),
                "d": _width(rng, 64, 2048 if f32 else 5120, 8), "D": min(D, 1024) if f32 else D,
                "dtype": "f32" if f32 else "bf16"}
    if kind == "lanczos":
        D = rng.choice([128, 256, 384, 512, 768, 1024, 1536, 2048])
        return {"kind": "lanczos", "N": _log(rng, 400, 32768), "d": 512, "D": D,
                "r": rng.choice([16, 24, 32, 48, 64]), "phi": rng.choice(["f32", "f32", "bf16"])}
    if kind == "windows":
        return {"kind": "windows", "B": rng.randint(1, 8), "N": _log(rng, 3000, 16384), "d": 512,
                "D": rng.choice([256, 512, 1024]), "r": rng.choice([16, 32]),
                "window": rng.choice([512, 1024, 2048])}
    if kind == "simhash":
        return {"kind": "simhash", "N": _log(rng, 500, 131072),
                "k": rng.choice([16, 24, 32, 48, 64]), "bits": rng.randint(6, 20)}
    f32 = rng.random() < 0.3
    return {"kind": "aggregate", "N": _log(rng, 300, 32768), "d": _width(rng, 64, 5120, 8),
            "dtype": "f32" if f32 else "bf16", "bits": rng.randint(8, 16),
            "rho": rng.choice([4.0, 8.0, 16.0]), "scheme": rng.choice(["max", "max", "median", "mean"])}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

TYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
SCHEMES = {"max": sls.POS_MAX, "median": sls.POS_MEDIAN, "mean": sls.POS_MEAN}
BACKENDS = {"global": sls.BACKEND_GLOBAL, "local": sls.BACKEND_LOCAL,
            "adaptive": sls.BACKEND_ADAPTIVE}
VOCAB = 32768
ZIPF = 1.1


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _randn(g, *shape, dtype=torch.float32):
    return torch.randn(*shape, generator=g, device=DEV, dtype=dtype)


def _ids(seed, N):
    """Zipf(1.1) token ids with 64-token spans copied from earlier positions
    until about a fifth of the tokens are copies."""
    rng = np.random.default_rng(seed)
    p = np.arange(1, VOCAB + 1, dtype=np.float64) ** -ZIPF
    cdf = np.cumsum(p)
    ids = np.searchsorted(cdf / cdf[-1], rng.random(N), side="right").clip(max=VOCAB - 1)
    for _ in range(N // 320):
        dst = int(rng.integers(64, N - 64))
        src = int(rng.integers(0, dst - 63))
        ids[dst:dst + 64] = ids[src:src + 64]
    return torch.from_numpy(ids.astype(np.int64)).to(DEV)


def _embed(g, ids, d, dtype):
    """Rows of a Gaussian table N(0, 1/d) for the ids that occur; float32
    embeddings carry N(0, 0.01) noise (no two tokens alike)."""
    uniq, inv = torch.unique(ids, return_inverse=True)
    X = (_randn(g, uniq.numel(), d) / math.sqrt(d))[inv]
    if dtype == "f32":
        X += 0.1 * _randn(g, *X.shape)
    return X.to(TYPES[dtype])


def _omega(g, D, d, dtype):
    W = (_randn(g, D, d) * d ** -0.25).to(TYPES[dtype])
    b = torch.rand(D, generator=g, device=DEV) * (2 * math.pi)
    return W, b


def _phi(g, ids, d, D):
    """Float32 features of bf16 embeddings, as the feature map gives them."""
    X = _embed(g, ids, d, "bf16").float()
    W, b = _omega(g, D, d, "bf16")
    W = W.float()
    phi = torch.empty((X.shape[0], D), device=DEV)
    for i in range(0, X.shape[0], 32768):
        phi[i:i + 32768] = math.sqrt(2.0 / D) * torch.cos(X[i:i + 32768] @ W.T + b)
    return phi


def _windows(case):
    """Rows of the windows of B prompts stored one after the other."""
    B, N, w = case["B"], case["N"], case["window"]
    row0 = [b * N + s for b in range(B) for s in range(0, N, w)]
    n = [min(w, N - s) for b in range(B) for s in range(0, N, w)]
    return row0, n


def _codes(g, ids, bits):
    """Codes as SimHash gives them: equal tokens share a code, and the leading
    directions are shared by many tokens, so cluster sizes are uneven."""
    uniq, inv = torch.unique(ids, return_inverse=True)
    k = 24
    U = _randn(g, uniq.numel(), k) * torch.linspace(2.0, 0.5, k, device=DEV)
    U[:, 0] += 1.0
    R = _randn(g, bits, k)
    bit = ((U @ R.T) > 0).to(torch.int64)
    code = (bit << torch.arange(bits, device=DEV)).sum(1)
    return code.to(torch.int32)[inv].contiguous()


def _config(case):
    return sls.Config.make(backend=BACKENDS[case["backend"]], rho=case["rho"], D=case["D"],
                           r=case["r"], bits=case["bits"], preserve_last=LAST,
                           window=case.get("window", 2048))


def prepare(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind in ("pass", "tokens"):
        B, N, d = case["B"], case["N"], case["d"]
        cfg = _config(case)
        W, b = _omega(g, case["D"], d, case["dtype"])
        st = {"cfg": cfg, "W": W, "b": b, "R": _randn(g, 32, case["r"]),
              "q1": _randn(g, B * N, dtype=torch.float64)}
        ids = torch.stack([_ids(seed * 1000 + k, N) for k in range(B)])
        if kind == "tokens":
            st["table"] = (_randn(g, case["V"], d) / math.sqrt(d)).to(TYPES[case["dtype"]])
            st["ids"] = ids[0].to(torch.int32)
            st["ws"] = sls.TokensWorkspace(cfg, TYPES[case["dtype"]], B, N, d, DEV)
        else:
            X = torch.empty((B, N, d), dtype=TYPES[case["dtype"]], device=DEV)
            for k in range(B):
                X[k] = _embed(g, ids[k], d, case["dtype"])
            st["X"] = X if B > 1 else X[0]
            st["q1"] = st["q1"].view(B, N) if B > 1 else st["q1"]
            st["ws"] = sls.Workspace(cfg, B, N, d, DEV)
        return {"kind": kind, **st}
    if kind == "features":
        X = _embed(g, _ids(seed, case["N"]), case["d"], case["dtype"])
        W, b = _omega(g, case["D"], case["d"], case["dtype"])
        return {"kind": kind, "X": X, "W": W, "b": b}
    if kind == "lanczos":
        phi = _phi(g, _ids(seed, case["N"]), case["d"], case["D"])
        if case["phi"] == "bf16":
            phi = phi.to(torch.bfloat16)
        return {"kind": kind, "phi": phi, "q1": _randn(g, case["N"], dtype=torch.float64),
                "r": case["r"]}
    if kind == "windows":
        ids = torch.cat([_ids(seed * 1000 + k, case["N"]) for k in range(case["B"])])
        row0, n = _windows(case)
        return {"kind": kind, "phi": _phi(g, ids, case["d"], case["D"]),
                "q1": _randn(g, ids.numel(), dtype=torch.float64), "r": case["r"],
                "row0": row0, "n": n}
    if kind == "simhash":
        return {"kind": kind, "U": _randn(g, case["N"], case["k"]) / math.sqrt(case["N"]),
                "R": _randn(g, 32, case["k"]), "bits": case["bits"]}
    if kind == "aggregate":
        ids = _ids(seed, case["N"])
        return {"kind": kind, "X": _embed(g, ids, case["d"], case["dtype"]),
                "codes": _codes(g, ids, case["bits"]), "M": math.ceil(case["N"] / case["rho"]),
                "scheme": SCHEMES[case["scheme"]]}
    raise ValueError(kind)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------


def run(st):
    kind = st["kind"]
    if kind == "pass":
        Xt, pos, t2m, _, _ = sls.compress(st["X"], st["cfg"], st["W"], st["b"], st["R"], st["q1"],
                                          workspace=st["ws"])
        return {"Xt": Xt, "pos": pos, "t2m": t2m}
    if kind == "tokens":
        Xt, pos, t2m, _, _ = sls.compress_tokens(st["ids"], st["table"], st["cfg"], st["W"],
                                                 st["b"], st["R"], st["q1"], workspace=st["ws"])
        return {"Xt": Xt, "pos": pos, "t2m": t2m}
    if kind == "features":
        return {"phi": sls.feature_map(st["X"], st["W"], st["b"])}
    if kind == "lanczos":
        theta, U, r_eff, alpha, beta = sls.lanczos_topr(st["phi"], st["q1"], st["r"])
        return {"theta": theta, "U": U, "r_eff": r_eff, "alpha": alpha, "beta": beta}
    if kind == "windows":
        theta, U, r_eff, alpha, beta = sls.lanczos_topr_batched(st["phi"], st["q1"], st["r"],
                                                                st["row0"], st["n"])
        return {"theta": theta, "U": U, "r_eff": r_eff, "alpha": alpha, "beta": beta}
    if kind == "simhash":
        return {"codes": sls.simhash(st["U"], st["R"], st["bits"])}
    Xt, pos, t2m = sls.aggregate(st["X"], st["codes"], st["M"], st["scheme"])
    return {"Xt": Xt, "pos": pos, "t2m": t2m}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------


def _lanczos_flops(n, D, r):
    # one product with Phi and one with its transpose per step, the
    # re-orthogonalisation, and U = Q S
    return 4.0 * n * D * r + 4.0 * n * r * r + 2.0 * n * r * r


def work(case):
    kind = case["kind"]
    esz = {"f32": 4, "bf16": 2}
    if kind in ("pass", "tokens"):
        B, N, d, D, r = case["B"], case["N"], case["d"], case["D"], case["r"]
        M = math.ceil((N - LAST) / case["rho"]) + LAST
        e = esz[case["dtype"]]
        rows = case["V"] if kind == "tokens" and case["V"] < N else B * N
        nb = rows * d * e + B * M * d * 4 + B * (M + N) * 4 + (N * 4 if kind == "tokens" else 0)
        if case["backend"] == "adaptive":  # every window on the chunk path
            return {"bytes": nb, "flops": 6.0 * B * N * d}
        nb += D * d * e + N * 8
        w = case.get("window", N)
        return {"bytes": nb, "flops": 2.0 * B * N * D * d + _lanczos_flops(B * N, D, min(r, w))}
    if kind == "features":
        N, d, D = case["N"], case["d"], case["D"]
        return {"bytes": (N + D) * d * esz[case["dtype"]] + N * D * 4.0 + 4 * D,
                "flops": 2.0 * N * d * D}
    if kind == "lanczos":
        N, D, r = case["N"], case["D"], case["r"]
        return {"bytes": N * D * float(esz[case["phi"]]) + N * 8 + N * r * 4,
                "flops": _lanczos_flops(N, D, r)}
    if kind == "windows":
        rows, D, r = case["B"] * case["N"], case["D"], case["r"]
        return {"bytes": rows * D * 4.0 + rows * 8 + rows * r * 4,
                "flops": _lanczos_flops(rows, D, r)}
    if kind == "simhash":
        N, k = case["N"], case["k"]
        return {"bytes": N * k * 4.0 + N * 4, "flops": 2.0 * N * k * case["bits"]}
    N, d = case["N"], case["d"]
    M = math.ceil(N / case["rho"])
    return {"bytes": N * d * float(esz[case["dtype"]]) + N * 4 + M * d * 4 + (M + N) * 4,
            "flops": 3.0 * N * d}


# ---------------------------------------------------------------------------
# float64 counterparts
# ---------------------------------------------------------------------------


def _lanczos64(phi, q1, r, tol=1e-10):
    """Algorithm 2 with two Gram-Schmidt passes, Eigh(T) and U = Q V, each
    eigenvector of T with a positive first entry."""
    phi = phi.double()
    n = phi.shape[0]
    Q = torch.zeros((r, n), dtype=torch.float64, device=DEV)
    a, b = np.zeros(r), np.zeros(r)
    Q[0] = q1 / q1.norm()
    k, scale = r, 0.0
    for j in range(r):
        z = phi @ (phi.T @ Q[j])
        alpha = torch.dot(Q[j], z)
        z = z - alpha * Q[j] - (b[j - 1] * Q[j - 1] if j else 0.0)
        for _ in range(2):
            z = z - Q[:j + 1].T @ (Q[:j + 1] @ z)
        a[j] = alpha.item()
        beta = z.norm().item()
        if j == r - 1:
            break
        scale = max(scale, abs(a[j]) + beta)
        if beta <= tol * scale:
            k = j + 1
            break
        b[j] = beta
        Q[j + 1] = z / beta
    T = np.diag(a[:k]) + np.diag(b[:k - 1], 1) + np.diag(b[:k - 1], -1)
    th, S = np.linalg.eigh(T)
    th, S = th[::-1], S[:, ::-1]
    S = S * np.where(S[0] < 0, -1.0, 1.0)
    theta = np.zeros(r)
    theta[:k] = th
    U = torch.zeros((n, r), dtype=torch.float64, device=DEV)
    U[:, :k] = Q[:k].T @ torch.from_numpy(S.copy()).to(DEV)
    return torch.from_numpy(theta).to(DEV), U, torch.from_numpy(a).to(DEV), torch.from_numpy(b).to(DEV)


def _groups(codes, M):
    """Members of the M groups: clusters of equal codes in code order, merged
    by rank or cut by D'Hondt seats (one guaranteed, ties to the lower code)."""
    codes = codes.cpu().numpy().view(np.uint32)
    order = np.argsort(codes, kind="stable")
    cut = np.flatnonzero(np.diff(codes[order])) + 1
    clusters = np.split(order, cut)
    C = len(clusters)
    if C >= M:
        lab = np.arange(C) * M // C
        return [np.sort(np.concatenate([clusters[t] for t in range(lo, hi)])) for lo, hi in
                zip(np.searchsorted(lab, np.arange(M)), np.searchsorted(lab, np.arange(M), "right"))]
    seats = np.ones(C, dtype=np.int64)
    heap = [(-len(c) / 2.0, t) for t, c in enumerate(clusters) if len(c) > 1]
    heapq.heapify(heap)
    for _ in range(M - C):
        _, t = heapq.heappop(heap)
        seats[t] += 1
        if seats[t] < len(clusters[t]):
            heapq.heappush(heap, (-len(clusters[t]) / (seats[t] + 1.0), t))
    return [p for c, s in zip(clusters, seats) for p in np.array_split(c, s)]


def _macro_tokens(X, groups):
    """The renormalised mean of each group, in float64."""
    lab = np.empty(X.shape[0], dtype=np.int64)
    for i, g in enumerate(groups):
        lab[g] = i
    lab = torch.from_numpy(lab).to(DEV)
    X = X.double()
    M = len(groups)
    cnt = torch.bincount(lab, minlength=M).double()
    mean = torch.zeros((M, X.shape[1]), dtype=torch.float64, device=DEV).index_add_(0, lab, X)
    mean /= cnt[:, None]
    eta = torch.zeros(M, dtype=torch.float64, device=DEV).index_add_(0, lab, X.norm(dim=1)) / cnt
    nrm = mean.norm(dim=1)
    scale = torch.where((cnt > 1) & (nrm >= 1e-30), eta / nrm.clamp(min=1e-300), 1.0)
    return mean * scale[:, None]


def _position(g, scheme):
    if scheme == sls.POS_MAX:
        return int(g.max())
    if scheme == sls.POS_MEDIAN:
        return int(np.sort(g)[(len(g) - 1) // 2])
    return int((2 * int(g.sum()) + len(g)) // (2 * len(g)))


def _chunk_window(X, m):
    """m consecutive groups of one window (numpy array_split sizes)."""
    return _macro_tokens(X, np.array_split(np.arange(X.shape[0]), m))


def _budgets(Nc, window, rho):
    """Macro-tokens per window: one each, the rest by largest remainder."""
    M, W = math.ceil(Nc / rho), -(-Nc // window)
    L = [window] * (W - 1) + [Nc - (W - 1) * window]
    E, den = M - W, Nc - W
    base = [E * (x - 1) // den if den else 0 for x in L]
    rem = [E * (x - 1) % den if den else 0 for x in L]
    for t in sorted(range(W), key=lambda i: (-rem[i], i))[:E - sum(base)]:
        base[t] += 1
    return L, [1 + x for x in base]


def _redundant(X, tau):
    X = X.double()
    s = X.sum(0)
    score = ((X / X.norm(dim=1, keepdim=True)).sum(0) @ s / (X.shape[0] * s.norm())).item()
    return score >= tau


def exact(case, seed):
    st = prepare(case, seed)
    kind = case["kind"]
    if kind == "features":
        X, W, b = st["X"].double(), st["W"].double(), st["b"].double()
        return {"phi": math.sqrt(2.0 / case["D"]) * torch.cos(X @ W.T + b)}
    if kind == "lanczos":
        th, U, a, b = _lanczos64(st["phi"], st["q1"], st["r"])
        return {"theta": th, "U": U, "r_eff": None, "alpha": a, "beta": b}
    if kind == "windows":
        got = [_lanczos64(st["phi"][r0:r0 + n], st["q1"][r0:r0 + n], st["r"])
               for r0, n in zip(st["row0"], st["n"])]
        return {"theta": torch.stack([x[0] for x in got]), "U": torch.cat([x[1] for x in got]),
                "r_eff": None, "alpha": torch.stack([x[2] for x in got]),
                "beta": torch.stack([x[3] for x in got])}
    if kind == "aggregate":
        groups = _groups(st["codes"], st["M"])
        key = [(_position(g, st["scheme"]), int(g.min())) for g in groups]
        order = sorted(range(len(groups)), key=lambda i: key[i])
        Xt = _macro_tokens(st["X"], [groups[i] for i in order])
        return {"Xt": Xt, "pos": None, "t2m": None}
    if kind == "pass" and case["backend"] == "adaptive":
        # the chunk path; None if the router sends a window elsewhere
        X = st["X"] if case["B"] > 1 else st["X"].unsqueeze(0)
        L, m = _budgets(case["N"] - LAST, case["window"], case["rho"])
        tau = min(0.70, max(0.55, 0.75 - 0.05 * math.log2(case["rho"])))
        out = []
        for k in range(case["B"]):
            rows, s = [], 0
            for n, mm in zip(L, m):
                if n > 4 and _redundant(X[k, s:s + n], tau):
                    return None
                rows.append(_chunk_window(X[k, s:s + n], mm))
                s += n
            out.append(torch.cat(rows + [X[k, s:].double()]))
        Xt = torch.stack(out)
        return {"Xt": Xt if case["B"] > 1 else Xt[0], "pos": None, "t2m": None}
    return None  # codes (whole values), and passes whose clusters rest on float32 signs


def tolerance(case):
    """About four times what was measured: the distance to exact() where there
    is one (features 6e-7: a sum of d float32 products; Ritz vectors 1.3e-7,
    their float32 output; macro-tokens 8e-8)."""
    kind = case["kind"]
    if kind == "simhash":
        return "exact"
    if kind == "features":
        return {"rel": 2.5e-6, "max": 1e-4}
    if kind in ("lanczos", "windows"):
        return {"rel": 6e-7, "max": 2e-5}
    if kind == "aggregate" or case["backend"] == "adaptive":
        return {"rel": 4e-7, "max": 1e-5}
    # a pass whose Lanczos sums ran in another order gave the same clusters on
    # all of eighteen prompts; room for a token whose code bit is a tie
    return {"rel": 0.02, "max": 0.9, "differ": 0.005}
