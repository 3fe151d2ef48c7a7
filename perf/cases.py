"""The calls whose speed counts: affinity propagation as a program uses this package.

Each case is one public call (or one whole clustering) on inputs shaped like
the package's own workloads: the 500- and 1000-point 2-D mixtures and the
2021 62-dimensional faces of the paper's tables, the 20000-point 64-D
mixture, the batches of image-like problems (200 to 4000 points, d = 4096)
and the 10^6-point landmark assignment.  Inputs come from a seed alone and
are made with torch, so they do not depend on the package's own arithmetic.
"""
import math

import numpy as np
import torch

from paper_0910_1650_gb300 import capi

DEV = "cuda"


def listed():
    return [
        # Algorithm 1 on the paper's small random 2-D sets: everything stays on the chip, latency counts
        {"name": "iterate_500", "op": "iterate", "n": 500, "d": 2, "k": 5, "damping": 0.9, "iters": 100},
        # ... on a mid-sized landmark set (Algorithm 3's landmarks), odd size
        {"name": "iterate_5003", "op": "iterate", "n": 5003, "d": 64, "k": 40, "damping": 0.9, "iters": 100},
        # ... on the 20000-point mixture: the headline sweep
        {"name": "iterate_20000", "op": "iterate", "n": 20000, "d": 64, "k": 50, "damping": 0.9, "iters": 100},
        # many independent problems of uneven sizes in one call
        {"name": "iterate_batch_48", "op": "iterate_batch", "count": 48, "lo": 200, "hi": 4000, "damping": 0.9,
         "iters": 50},
        # a whole clustering of the paper's face-sized set: similarity, messages to convergence, labels
        {"name": "cluster_2021", "op": "cluster", "n": 2021, "d": 62, "k": 86, "damping": 0.9},
        # the similarity build at its smallest, with tie-break noise
        {"name": "similarity_fp32_1000", "op": "similarity", "n": 1000, "d": 2, "k": 5, "precision": "fp32",
         "pref": "median", "noise": 1e-12},
        # ... the default precision on subspace-like features
        {"name": "similarity_fp32_10000", "op": "similarity", "n": 10000, "d": 100, "k": 10, "precision": "fp32",
         "pref": "median", "noise": 0.0},
        # ... the tensor-core build of the headline workload
        {"name": "similarity_bf16_20000", "op": "similarity", "n": 20000, "d": 64, "k": 50, "precision": "bf16",
         "pref": "median", "noise": 0.0},
        # the similarity build of a batch of image problems
        {"name": "similarity_batch_32", "op": "similarity_batch", "count": 32, "lo": 200, "hi": 4000, "d": 4096},
        # Algorithm 3 Step 2: a million points to their nearest of a thousand exemplars
        {"name": "assign_1000000", "op": "assign", "n": 1000000, "d": 128, "c": 1000, "best": True},
        # one Adam step of the warm-start network at the training loop's batch size
        {"name": "train_4096", "op": "train", "rows": 4096},
        # the learned warm start of a batch (features, forward pass, messages)
        {"name": "warm_start_48", "op": "warm_start", "count": 48, "lo": 200, "hi": 4000},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["iterate", "iterate", "iterate_batch", "cluster", "similarity", "similarity",
                     "similarity_batch", "assign", "train", "warm_start"])
    if op == "iterate":
        n = _log(rng, 100, 20000)
        return {"op": op, "n": n, "d": rng.choice([2, 64]), "k": rng.randint(5, 50), "damping": 0.9,
                "iters": rng.choice([50, 100])}
    if op == "iterate_batch":
        return {"op": op, "count": rng.randint(4, 48), "lo": rng.choice([100, 200]),
                "hi": rng.randint(500, 4000), "damping": 0.9, "iters": 50}
    if op == "cluster":
        return {"op": op, "n": _log(rng, 300, 3000), "d": rng.randint(40, 80), "k": rng.randint(20, 90),
                "damping": 0.9}
    if op == "similarity":
        precision = rng.choice(["fp32", "bf16"])
        n = _log(rng, 100, 20000 if precision == "bf16" else 10000)
        if precision == "bf16":
            d = rng.choice([2, 64, 100, 128, 300] if n > 8000 else [2, 64, 100, 128, 300, 1000, 4096])
        else:
            d = rng.choice([2, 62, 64, 100] if n > 3000 else [2, 62, 100, 128, 300, 1000])
        return {"op": op, "n": n, "d": d, "k": rng.randint(5, 50), "precision": precision,
                "pref": rng.choice(["median", "median", "scalar", "vector"]),
                "noise": rng.choice([0.0, 0.0, 1e-12])}
    if op == "similarity_batch":
        return {"op": op, "count": rng.randint(2, 32), "lo": 200, "hi": rng.randint(500, 4000),
                "d": rng.choice([32, 300, 4096])}
    if op == "assign":
        n = _log(rng, 10000, 1000000)
        return {"op": op, "n": n, "d": rng.choice([16, 64, 100, 128]), "c": min(n // 8, _log(rng, 50, 1000)),
                "best": rng.choice([True, False])}
    if op == "train":
        return {"op": op, "rows": rng.randint(64, 4096)}
    return {"op": op, "count": rng.randint(2, 48), "lo": 200, "hi": rng.randint(500, 4000)}


# ---- inputs ---------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1000003 + 17)
    return g


def _mixture(g, n, d, k):
    """Points of k Gaussians: in the plane (centres in a box, sigma 1) or in d dimensions."""
    if d == 2:
        centres = torch.rand(k, d, generator=g, device=DEV) * 20 - 10
    else:
        centres = torch.randn(k, d, generator=g, device=DEV) * 5
    labels = torch.randint(0, k, (n,), generator=g, device=DEV)
    return centres[labels] + torch.randn(n, d, generator=g, device=DEV)


def _sizes(case):
    """The problem sizes of a batch: uniform in [lo, hi], the same for every seed."""
    r = np.random.RandomState(case["count"] * 7919 + case["lo"] + case["hi"])
    return [int(x) for x in r.randint(case["lo"], case["hi"] + 1, size=case["count"])]


def _distances(X, chunk=4096):
    """-|x_i - x_k|^2 in 64 bits, zero on the diagonal."""
    X = X.double()
    X = X - X.mean(0)
    n = X.shape[0]
    nrm = (X * X).sum(1)
    S = torch.empty(n, n, dtype=torch.float64, device=X.device)
    for lo in range(0, n, chunk):
        hi = min(n, lo + chunk)
        S[lo:hi] = (2 * (X[lo:hi] @ X.T) - nrm[lo:hi, None] - nrm[None, :]).clamp_(max=0)
    S.diagonal().zero_()
    return S


def _square(n):
    return capi.empty_square(n, DEV, 0.0)


def _similarities(g, n, d, k):
    """A float32 similarity matrix with a common preference near the median."""
    S64 = _distances(_mixture(g, n, d, k))
    m = min(n, 1000)
    p = S64[:m, :m][~torch.eye(m, dtype=torch.bool, device=DEV)].median()
    S = _square(n)
    S.copy_(S64)
    S.diagonal().fill_(float(p))
    return S, float(p)


def _arena(sizes):
    ld = [capi.padded_ld(n) for n in sizes]
    off, at = [], 0
    for n, l in zip(sizes, ld):
        off.append(at)
        at += n * l
    return off, ld, at


def _view(T, off, n, ld):
    return T[off:off + n * ld].view(n, ld)[:, :n]


def _batch(seed, case):
    """S of every problem of a batch in one arena, and each problem's preference."""
    g = _gen(seed)
    sizes = _sizes(case)
    off, ld, total = _arena(sizes)
    S = torch.zeros(total, dtype=torch.float32, device=DEV)
    prefs = []
    for n, o, l in zip(sizes, off, ld):
        Sb, p = _similarities(g, n, 32, 5 + n % 36)
        _view(S, o, n, l).copy_(Sb)
        prefs.append(p)
    return sizes, off, ld, S, prefs


def _images(g, n, d):
    """Nonnegative image-like vectors: rank-20 templates and uniform noise."""
    k = 5 + n % 36
    T = torch.rand(k, 20, generator=g, device=DEV) @ torch.rand(20, d, generator=g, device=DEV)
    T = T / T.amax(1, keepdim=True)
    labels = torch.randint(0, k, (n,), generator=g, device=DEV)
    return (T[labels] + 0.05 * torch.rand(n, d, generator=g, device=DEV)).clamp_(0, 1)


def _network(g):
    """Weights of the warm-start network (25-256-256-3) with a standardised input."""
    parts = []
    for o, i in ((256, 25), (256, 256), (3, 256)):
        parts += [torch.randn(o * i, generator=g, device=DEV) * math.sqrt(2.0 / i),
                  torch.randn(o, generator=g, device=DEV) * 0.05]
    parts += [torch.randn(25, generator=g, device=DEV) * 0.1, 0.5 + torch.rand(25, generator=g, device=DEV)]
    P = torch.cat(parts)
    return P, P.to(torch.bfloat16)


def _unpack(P):
    out, at = [], 0
    for shape in ((256, 25), (256,), (256, 256), (256,), (3, 256), (3,), (25,), (25,)):
        n = int(np.prod(shape))
        out.append(P[at:at + n].view(*shape))
        at += n
    return out


# ---- one case: inputs, the call, its work and its exact answer -------------------------

def prepare(case, seed):
    g, op = _gen(seed), case["op"]
    if op == "iterate":
        S, _ = _similarities(g, case["n"], case["d"], case["k"])
        return {"case": case, "S": S, "R": _square(case["n"]), "A": _square(case["n"])}
    if op == "iterate_batch":
        sizes, off, ld, S, _ = _batch(seed, case)
        return {"case": case, "n": sizes, "off": off, "ld": ld, "S": S, "R": torch.zeros_like(S),
                "A": torch.zeros_like(S), "ws": capi.ap_iterate_batched_workspace(sizes, ld, DEV)}
    if op == "cluster":
        n = case["n"]
        return {"case": case, "X": _mixture(g, n, case["d"], case["k"]), "S": _square(n), "R": _square(n),
                "A": _square(n)}
    if op == "similarity":
        n = case["n"]
        X = _mixture(g, n, case["d"], case["k"])
        pref = {"median": "median", "scalar": -7.5,
                "vector": -torch.rand(n, generator=g, device=DEV) * 10 - 1}[case["pref"]]
        return {"case": case, "X": X, "S": _square(n), "pref": pref}
    if op == "similarity_batch":
        sizes = _sizes(case)
        d = case["d"]
        off, ld, total = _arena(sizes)
        X = torch.cat([_images(g, n, d) for n in sizes])
        xoff = [int(x) * d for x in np.concatenate([[0], np.cumsum(sizes)[:-1]])]
        return {"case": case, "n": sizes, "off": off, "ld": ld, "xoff": xoff, "X": X,
                "S": torch.zeros(total, dtype=torch.float32, device=DEV),
                "ws": capi.ap_similarity_batched_workspace(sizes, d, DEV)}
    if op == "assign":
        n, d, c = case["n"], case["d"], case["c"]
        centres = torch.randn(c, d, generator=g, device=DEV) * 4
        labels = torch.randint(0, c, (n,), generator=g, device=DEV)
        X = torch.randn(n, d, generator=g, device=DEV).mul_(0.5).add_(centres[labels])
        picks = torch.randperm(n, generator=g, device=DEV)[:c].sort().values.int()
        return {"case": case, "X": X, "centres": picks}
    if op == "train":
        rows = case["rows"]
        P, P16 = _network(g)
        F = torch.randn(rows, 25, generator=g, device=DEV)
        T = torch.randn(rows, 3, generator=g, device=DEV)
        T[:, 2] = (T[:, 2] > 1).float()
        M = torch.randn(P.numel(), generator=g, device=DEV) * 1e-3
        V = torch.rand(P.numel(), generator=g, device=DEV) * 1e-6 + 1e-7
        M[-50:] = 0
        V[-50:] = 0
        return {"case": case, "P": P, "P16": P16, "M": M, "V": V, "F": F, "T": T,
                "ws": capi.workspace(capi.lib().apl_workspace_size(rows), DEV)}
    sizes, off, ld, S, prefs = _batch(seed, case)
    P, P16 = _network(g)
    return {"case": case, "n": sizes, "off": off, "ld": ld, "S": S, "R": torch.zeros_like(S),
            "A": torch.zeros_like(S), "scale": [abs(p) for p in prefs], "P": P, "P16": P16,
            "Y": torch.zeros(sum(sizes), 3, device=DEV), "ws": capi.apl_warm_start_batched_workspace(sizes, DEV)}


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "iterate":
        R, A, res, dec = capi.ap_iterate(s["S"], s["R"], s["A"], damping=case["damping"],
                                         max_iter=case["iters"], conv_iter=0, cold=True)
        return {"R": R, "A": A, "decisions": dec, "iters": res["iters"]}
    if op == "iterate_batch":
        res, _ = capi.ap_iterate_batched(s["S"], s["R"], s["A"], s["off"], s["n"], s["ld"],
                                         damping=case["damping"], max_iter=case["iters"], conv_iter=0,
                                         ws=s["ws"], cold=True)
        return {"R": s["R"], "A": s["A"], "iters": sum(r["iters"] for r in res)}
    if op == "cluster":
        S, p = capi.ap_similarity(s["X"], s["S"])
        R, A, res, _ = capi.ap_iterate(S, s["R"], s["A"], damping=case["damping"], max_iter=1000, conv_iter=15,
                                       cold=True)
        idx, ex = capi.ap_exemplars(S, R, A)
        return {"S": S, "R": R, "A": A, "idx": idx, "preference": p, "dpsim": ex["dpsim"],
                "netsim": ex["netsim"]}
    if op == "similarity":
        S, p = capi.ap_similarity(s["X"], s["S"], precision=case["precision"], pref=s["pref"],
                                  noise_rel=case["noise"], seed=9)
        return {"S": S, "preference": p}
    if op == "similarity_batch":
        prefs = capi.ap_similarity_batched(s["X"], s["xoff"], s["n"], s["S"], s["off"], s["ld"], ws=s["ws"])
        return {"S": s["S"], "preferences": np.array(prefs, dtype=np.float32)}
    if op == "assign":
        out = capi.lap_assign(s["X"], s["centres"], best=case["best"])
        return {"idx": out[0], "best": out[1]} if case["best"] else {"idx": out}
    if op == "train":
        loss, grad = capi.apl_train_step(s["P"], s["P16"], s["M"], s["V"], 100, 1e-3, s["F"], s["T"],
                                         ws=s["ws"], want_grad=True)
        return {"P": s["P"], "P16": s["P16"], "M": s["M"], "V": s["V"], "loss": loss, "grad": grad}
    R, A = capi.apl_warm_start_batched(s["S"], s["R"], s["A"], s["off"], s["n"], s["ld"], s["scale"], s["P"],
                                       s["P16"], Y=s["Y"], ws=s["ws"])
    return {"R": R, "A": A, "Y": s["Y"]}


def _message_work(sum_n2, iters):
    """S read and R, A written once where the three matrices fit on the chip, each iteration's 20 bytes an
    entry (S, R, A read, R, A written) where they do not; about ten operations an entry and iteration."""
    on_chip = 12.0 * sum_n2 <= 129e6
    return {"bytes": 12.0 * sum_n2 if on_chip else 20.0 * sum_n2 * iters, "flops": 10.0 * sum_n2 * iters}


def _mean_n2(case):
    lo, hi = case["lo"], case["hi"]
    return (hi ** 3 - lo ** 3) / (3.0 * max(hi - lo, 1))


def work(case):
    op = case["op"]
    if op == "iterate":
        return _message_work(float(case["n"]) ** 2, case["iters"])
    if op == "iterate_batch":
        return _message_work(case["count"] * _mean_n2(case), case["iters"])
    if op == "cluster":
        n, d = float(case["n"]), case["d"]
        w = _message_work(n * n, 60)        # about 60 iterations to convergence
        return {"bytes": w["bytes"] + 4 * n * d, "flops": w["flops"] + n * n * d}
    if op == "similarity":
        n, d = float(case["n"]), case["d"]
        return {"bytes": 4 * n * n + 4 * n * d, "flops": n * n * d}      # a symmetric product
    if op == "similarity_batch":
        n2, rows = case["count"] * _mean_n2(case), case["count"] * 0.5 * (case["lo"] + case["hi"])
        return {"bytes": 4 * n2 + 4 * rows * case["d"], "flops": n2 * case["d"]}
    if op == "assign":
        n, d, c = float(case["n"]), case["d"], case["c"]
        return {"bytes": 4 * n * d + (8 if case["best"] else 4) * n, "flops": 2 * n * d * c}
    if op == "train":
        rows, weights = float(case["rows"]), 25 * 256 + 256 * 256 + 3 * 256
        return {"bytes": 4 * 28 * rows + 4 * 8 * weights, "flops": 6 * rows * weights}
    n2, rows = case["count"] * _mean_n2(case), case["count"] * 0.5 * (case["lo"] + case["hi"])
    return {"bytes": 12 * n2, "flops": 2 * rows * (25 * 256 + 256 * 256 + 3 * 256)}


# ---- 64-bit answers -------------------------------------------------------------------

def _median(S):
    """The median of the off-diagonal entries (the mean of the middle two) by bisection."""
    n = S.shape[0]
    m = n * (n - 1)
    D = S.clone()
    D.diagonal().fill_(math.inf)
    found = []
    for rank in ((m - 1) // 2, m // 2):
        lo, hi = float(S.min()) - 1.0, 1.0              # count(<= lo) <= rank < count(<= hi)
        for _ in range(70):
            mid = 0.5 * (lo + hi)
            if int((D <= mid).sum()) > rank:
                hi = mid
            else:
                lo = mid
        found.append(hi)
    return 0.5 * (found[0] + found[1])


def _rounded(X):
    """Features as the tensor-core path defines them: centred on their mean, then bf16."""
    mean = X.double().mean(0).float()
    return (X - mean).to(torch.bfloat16)


def _similarity64(X, precision):
    if precision == "fp32":
        return _distances(X)
    B = _rounded(X).double()
    nrm = (B * B).sum(1)
    S = (2 * (B @ B.T) - nrm[:, None] - nrm[None, :]).clamp_(max=0)
    S.diagonal().zero_()
    return S


def _messages(S, lam, max_iter, conv_iter):
    """Algorithm 1 from R = A = 0 in the precision of S."""
    n = S.shape[0]
    R, A = torch.zeros_like(S), torch.zeros_like(S)
    rows = torch.arange(n, device=S.device)
    before, same = None, 0
    for _ in range(max_iter):
        V = A + S
        m1, j1 = V.max(1)
        V[rows, j1] = -math.inf
        m2 = V.max(1).values
        V = S - m1[:, None]
        V[rows, j1] = S[rows, j1] - m2
        R.mul_(lam).add_(V, alpha=1 - lam)
        P = R.clamp(min=0)
        P.diagonal().zero_()
        colp = P.sum(0)
        torch.sub(colp + R.diagonal(), P, out=V)
        V.clamp_(max=0)
        V.diagonal().copy_(colp)
        A.mul_(lam).add_(V, alpha=1 - lam)
        if conv_iter:
            E = (A + R).argmax(1) == rows
            same = same + 1 if before is not None and torch.equal(E, before) else 1
            before = E
            if same >= conv_iter and bool(E.any()):
                break
    return R, A


def exact(case, seed):
    op = case["op"]
    s = prepare(case, seed)
    if op == "iterate":
        R, A = _messages(s["S"].double(), case["damping"], case["iters"], 0)
        return {"R": R, "A": A, "decisions": None, "iters": None}
    if op in ("iterate_batch", "warm_start"):
        R, A = torch.zeros_like(s["S"], dtype=torch.float64), torch.zeros_like(s["S"], dtype=torch.float64)
        if op == "iterate_batch":
            for n, o, l in zip(s["n"], s["off"], s["ld"]):
                r, a = _messages(_view(s["S"], o, n, l).double(), case["damping"], case["iters"], 0)
                _view(R, o, n, l).copy_(r)
                _view(A, o, n, l).copy_(a)
            return {"R": R, "A": A, "iters": None}
        Y = []
        for n, o, l, scale in zip(s["n"], s["off"], s["ld"], s["scale"]):
            y = _forward(s["P"], s["P16"], _features(_view(s["S"], o, n, l), scale))[-1]
            a = _view(A, o, n, l)
            a.copy_((y[:, 0] * scale).clamp(max=0).expand(n, n))
            a.diagonal().copy_((y[:, 1] * scale).clamp(min=0))
            Y.append(y)
        return {"R": R, "A": A, "Y": torch.cat(Y)}
    if op == "cluster":
        S = _distances(s["X"])
        p = _median(S)
        S.diagonal().fill_(p)
        R, A = _messages(S, case["damping"], 1000, 15)
        ex = torch.nonzero((A + R).argmax(1) == torch.arange(case["n"], device=DEV))[:, 0]
        dp = S[:, ex].max(1).values
        dp[ex] = 0
        return {"S": S, "R": R, "A": A, "idx": None, "preference": p, "dpsim": float(dp.sum()),
                "netsim": float(dp.sum() + p * ex.numel())}
    if op == "similarity":
        S = _similarity64(s["X"], case["precision"])
        p = {"median": lambda: _median(S), "scalar": lambda: -7.5, "vector": lambda: math.nan}[case["pref"]]()
        S.diagonal().copy_(s["pref"]) if case["pref"] == "vector" else S.diagonal().fill_(p)
        return {"S": S, "preference": p}
    if op == "similarity_batch":
        S, prefs, at = torch.zeros_like(s["S"], dtype=torch.float64), [], 0
        for n, o, l in zip(s["n"], s["off"], s["ld"]):
            Sb = _similarity64(s["X"][at:at + n], "bf16")
            at += n
            prefs.append(_median(Sb))
            Sb.diagonal().fill_(prefs[-1])
            _view(S, o, n, l).copy_(Sb)
        return {"S": S, "preferences": np.array(prefs)}
    if op == "assign":
        if not case["best"]:
            return None
        B = _rounded(s["X"])
        E = B[s["centres"].long()].double()
        nrm = (E * E).sum(1)
        best = torch.cat([(2 * (B[lo:lo + 65536].double() @ E.T) - nrm).max(1).values
                          for lo in range(0, case["n"], 65536)])
        return {"idx": None, "best": best}
    return _train64(s, 100, 1e-3)


def _features(S, scale):
    n = S.shape[0]
    D = S.double().clone()
    D.diagonal().fill_(-math.inf)
    top, nbr = D.sort(dim=1, descending=True, stable=True)
    top, nbr = top[:, :16], nbr[:, :16]
    off = D.masked_fill(torch.isinf(D), 0.0)
    mean = off.sum(1) / (n - 1)
    std = (((off - mean[:, None]) ** 2).sum(1) - mean ** 2).clamp(min=0).div(n - 1).sqrt()
    counts = [torch.log1p((D >= -(scale * q)).sum(1).double()) for q in (0.125, 0.25, 0.5, 1.0)]
    dens = counts[1]
    near = dens[nbr]
    F = torch.cat([top / scale, torch.stack([mean / scale, std / scale, S.diagonal().double() / scale, *counts,
                                             dens - near.max(1).values,
                                             (near > dens[:, None]).double().mean(1)], 1)], 1)
    return F


def _forward(P, P16, F):
    W1, _, W2, _, W3, _, _, _ = _unpack(P16.double())
    _, b1, _, b2, _, b3, mu, isd = _unpack(P.double())
    X = (F.double() - mu) * isd
    H1 = (X @ W1.T + b1).clamp(min=0)
    H2 = (H1 @ W2.T + b2).clamp(min=0)
    return X, H1, H2, H2 @ W3.T + b3


def _train64(s, step, lr):
    P, T, rows = s["P"].double(), s["T"].double(), s["F"].shape[0]
    _, _, W2, _, W3, _, _, _ = _unpack(s["P16"].double())
    X, H1, H2, Y = _forward(s["P"], s["P16"], s["F"])
    d, z = Y[:, :2] - T[:, :2], Y[:, 2]
    loss = (d * d).sum(1) + torch.nn.functional.softplus(z) - T[:, 2] * z
    G3 = torch.cat([2 * d, (torch.sigmoid(z) - T[:, 2])[:, None]], 1) / rows
    G2 = (G3 @ W3) * (H2 > 0)
    G1 = (G2 @ W2) * (H1 > 0)
    grad = torch.cat([(G1.T @ X).reshape(-1), G1.sum(0), (G2.T @ H1).reshape(-1), G2.sum(0),
                      (G3.T @ H2).reshape(-1), G3.sum(0), torch.zeros(50, dtype=torch.float64, device=DEV)])
    M = 0.9 * s["M"].double() + 0.1 * grad
    V = 0.999 * s["V"].double() + 0.001 * grad * grad
    P = P - lr * (M / (1 - 0.9 ** step)) / ((V / (1 - 0.999 ** step)).sqrt() + 1e-8)
    return {"P": P, "P16": P, "M": M, "V": V, "loss": loss.mean().reshape(1), "grad": grad}
