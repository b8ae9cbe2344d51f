"""The framework's work, as measurable cases: whole calls through the public binding.

Every case is one pass of something a user of ``paper_2303_05455_gb300.ivhd`` does:

* ``embed``    one whole embedding of a kNN graph: create (random neighbours, layout, initial
               positions), the steps, positions read back; with ``report`` > 0 the stress is
               asked for every ``report`` steps, as the optimiser curves do.
* ``batch``    several embeddings in one context (``Embedding.batch``), same pass.
* ``knn``      the exact kNN graph of a feature matrix.
* ``query``    arriving points: exact neighbours in a held base set, and their placement.
* ``train``    one epoch of the placement network from its initial weights (Adam steps).
* ``place``    the placement network applied to new rows.
* ``quality``  Q_NX and cf_nn of an embedding on sampled rows.

Sizes are those of the benchmark workloads (``synth.WORKLOADS``, ``synth.batch_workload``,
``bench_warmstart``) and odd ones between them.  Inputs are drawn on the GPU from the seed:
kNN-shaped graphs with clusters and the skewed in-degrees of high-dimensional kNN graphs,
Gaussian mixtures (float rows) and prototype images with noise (uint8 rows).
"""
import math

import numpy as np
import torch

from paper_2303_05455_gb300 import ivhd

DEV = "cuda"


# ---- the cases ----------------------------------------------------------------


def _embed(M, k, r, steps, opt="momentum", b=0.001, pos="f32", report=0):
    return {"kind": "embed", "M": M, "k": k, "r": r, "steps": steps, "opt": opt, "b": b,
            "pos": pos, "report": report}


def listed():
    return [
        # the small workload: 2,000 points, where launches and latency are the time
        dict(_embed(2000, 2, 1, 1000, b=0.01), name="embed_2k"),
        # an interactive mid-size run with a stress report every 50 steps, odd size, Nesterov
        dict(_embed(20011, 3, 2, 500, opt="nesterov", report=50), name="embed_20k_nesterov_report"),
        # the 70,000-image workload
        dict(_embed(70000, 5, 1, 2000), name="embed_70k"),
        # a larger odd size with half-precision gathers and the third optimiser's neighbours k = 10
        dict(_embed(300007, 10, 1, 300, pos="f16"), name="embed_300k_k10_f16"),
        # the headline workload: 1.4e6 points, 2,000 steps
        dict(_embed(1400000, 5, 1, 2000), name="embed_1400k"),
        # many embeddings at once: sizes log-uniform in [5,000, 200,000], as the batch benchmark
        {"name": "batch_16", "kind": "batch", "n": 16, "lo": 5000, "hi": 200000, "steps": 500},
        # graph construction: float features (100 dimensions) and images (784 bytes)
        {"name": "knn_f32_300k", "kind": "knn", "dtype": "f32", "M": 300000, "N": 100, "k": 5},
        {"name": "knn_u8_70k", "kind": "knn", "dtype": "u8", "M": 70000, "N": 784, "k": 5},
        # a batch of 10,000 arriving images placed by its nearest neighbour among 200,000
        {"name": "query_u8_10k", "kind": "query", "dtype": "u8", "M": 200000, "Mq": 10000,
         "N": 784, "k": 1},
        # the placement network: one epoch of 200,000 images in batches of 4,096 ...
        {"name": "train_epoch", "kind": "train", "n_in": 784, "hidden": 512, "batch": 4096,
         "batches": 48},
        # ... and its use on the 1.4e6-point held-out set
        {"name": "place_1400k", "kind": "place", "dtype": "u8", "n": 1400000, "n_in": 784,
         "hidden": 512},
        # quality of a 70,000-point embedding over all its rows
        {"name": "quality_70k", "kind": "quality", "M": 70000, "rows": 70000, "k": 5, "nn": 10},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["embed", "embed", "embed", "batch", "knn", "knn", "query", "train", "place",
                       "place", "quality"])
    if kind == "embed":
        M = _log(rng, 1000, 1000000)
        k = rng.choice([2, 3, 5, 7, 10])
        opt = rng.choice(["momentum", "momentum", "nesterov", "adadelta"])
        pos = "f32" if opt == "adadelta" else rng.choice(["f32", "f32", "f16", "bf16"])
        b = 0.01 if M < 5000 and k <= 3 else 0.001
        # Adadelta grows its steps (and with them rounding differences): short runs
        steps = rng.randint(60, 200) if opt == "adadelta" else _log(rng, 100, 1500)
        return _embed(M, k, rng.choice([1, 1, 2]), steps, opt, b, pos, rng.choice([0, 0, 50, 97]))
    if kind == "batch":
        return {"kind": "batch", "n": rng.randint(2, 20), "lo": 1000, "hi": _log(rng, 5000, 150000),
                "steps": _log(rng, 64, 500)}
    if kind == "knn":
        dtype = rng.choice(["f32", "u8"])
        return {"kind": "knn", "dtype": dtype, "M": _log(rng, 1000, 150000),
                "N": _log(rng, 8, 200) if dtype == "f32" else _log(rng, 64, 1000),
                "k": rng.choice([1, 2, 3, 5, 8, 10, 15, 20])}
    if kind == "query":
        dtype = rng.choice(["f32", "u8"])
        return {"kind": "query", "dtype": dtype, "M": _log(rng, 2000, 200000),
                "Mq": _log(rng, 16, 20000),
                "N": _log(rng, 8, 200) if dtype == "f32" else _log(rng, 64, 800),
                "k": rng.choice([1, 1, 3, 5, 10])}
    if kind == "train":
        return {"kind": "train", "n_in": 8 * rng.randint(4, 110), "hidden": 16 * rng.randint(4, 40),
                "batch": 8 * _log(rng, 8, 768), "batches": rng.randint(4, 40)}
    if kind == "place":
        return {"kind": "place", "dtype": rng.choice(["u8", "u8", "f32", "bf16"]),
                "n": _log(rng, 1, 700000), "n_in": 8 * rng.randint(4, 110),
                "hidden": rng.choice([512, 512, 16 * rng.randint(4, 40)])}
    M = _log(rng, 1000, 300000)
    return {"kind": "quality", "M": M, "rows": min(M, _log(rng, 500, 20000)),
            "k": rng.choice([2, 5, 10]), "nn": rng.choice([2, 10, 100])}


# ---- inputs ---------------------------------------------------------------------


def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + salt * 7919 + 12345) & 0x7FFFFFFFFFFF)
    return g


def _sizes(M):
    """Cluster sizes: equal below 100,000 points, a power law (exponent 1.5, 50 clusters) above."""
    if M < 100000:
        C = max(2, min(50, M // 200))
        s = np.full(C, M // C, dtype=np.int64)
        s[: M - int(s.sum())] += 1
        return s
    w = np.arange(1, 51, dtype=np.float64) ** -1.5
    s = np.floor(w / w.sum() * M).astype(np.int64)
    s[0] += M - int(s.sum())
    return s


def _labels(M, g):
    lab = torch.repeat_interleave(torch.arange(len(_sizes(M)), device=DEV),
                                  torch.from_numpy(_sizes(M)).to(DEV))
    return lab[torch.randperm(M, generator=g, device=DEV)]


def _graph(M, k, g):
    """kNN-shaped rows (k distinct ids, never the row's own): neighbours inside the row's
    cluster, drawn by a log-normal popularity, so that in-degrees are skewed as those of
    high-dimensional kNN graphs (median about a third of the mean, hubs of several hundred)."""
    lab = _labels(M, g)
    members = torch.argsort(lab, stable=True)
    w = torch.exp(1.5 * torch.randn(M, generator=g, device=DEV, dtype=torch.float64)).clamp(max=600)
    cum = torch.cumsum(w[members], 0)
    ends = torch.from_numpy(np.cumsum(_sizes(M))).to(DEV)
    hi = cum[ends - 1]
    lo = torch.cat([torch.zeros(1, device=DEV, dtype=torch.float64), hi[:-1]])

    def pick(rows):
        c = lab[rows]
        u = torch.rand(rows.numel(), generator=g, device=DEV, dtype=torch.float64)
        at = torch.searchsorted(cum, lo[c] + u * (hi[c] - lo[c]), right=True).clamp(max=M - 1)
        return members[at]

    own = torch.arange(M, device=DEV)
    out = torch.stack([pick(own) for _ in range(k)], 1)
    while True:
        bad = out == own[:, None]
        for s in range(1, k):
            bad[:, s] |= (out[:, :s] == out[:, s:s + 1]).any(1)
        r, s = bad.nonzero(as_tuple=True)
        if r.numel() == 0:
            return out.to(torch.int32).contiguous(), lab
        out[r, s] = pick(r)


def _rows(dtype, M, N, seed, salt):
    """Feature rows and labels; the mixture (centres or prototypes) depends on the seed only."""
    gc, g = _gen(seed, 1), _gen(seed, salt)
    C = 10 if dtype == "u8" else 20
    lab = torch.randint(0, C, (M,), generator=g, device=DEV)
    if dtype == "u8":
        centre = torch.randint(0, 256, (C, N), generator=gc, device=DEV).float()
        out = torch.empty((M, N), dtype=torch.uint8, device=DEV)
        scale = 40.0
    else:
        centre = 5 * torch.randn((C, N), generator=gc, device=DEV)
        out = torch.empty((M, N), dtype=torch.float32, device=DEV)
        scale = 1.0
    step = max(1, (1 << 27) // N)
    for s in range(0, M, step):
        e = min(M, s + step)
        x = centre[lab[s:e]] + scale * torch.randn((e - s, N), generator=g, device=DEV)
        out[s:e] = x.round().clamp(0, 255).to(torch.uint8) if dtype == "u8" else x
    return out, lab


def _batch_shapes(case, seed):
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    out = []
    for _ in range(case["n"]):
        M = int(round(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"])))))
        out.append((M, int(rng.choice([2, 3, 5, 10])), int(rng.choice([1, 2]))))
    return out


def _net_params(n_in, hidden, seed):
    rng = np.random.Generator(np.random.PCG64(int(seed) + 17))
    parts = []
    for fo, fi, sc in ((hidden, n_in, 1.0), (hidden, hidden, 1.0), (2, hidden, 0.1)):
        lim = math.sqrt(6.0 / fi)
        parts += [rng.uniform(-lim, lim, fo * fi) * sc, rng.uniform(-0.05, 0.05, fo)]
    return torch.from_numpy(np.concatenate(parts).astype(np.float32)).to(DEV)


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "seed": int(seed)}
    if kind == "embed":
        st["knn"], _ = _graph(case["M"], case["k"], _gen(seed))
    elif kind == "batch":
        # the mix of sizes is the case's own; graphs and streams are the seed's
        st["shapes"] = _batch_shapes(case, 64)
        st["graphs"] = [_graph(M, k, _gen(seed, e))[0] for e, (M, k, _) in enumerate(st["shapes"])]
    elif kind == "knn":
        st["X"], _ = _rows(case["dtype"], case["M"], case["N"], seed, 2)
    elif kind == "query":
        X, lab = _rows(case["dtype"], case["M"], case["N"], seed, 2)
        st["X"] = X
        st["Q"], _ = _rows(case["dtype"], case["Mq"], case["N"], seed, 3)
        g = _gen(seed, 4)
        st["Y"] = (10 * torch.rand((20, 2), generator=g, device=DEV)[lab]
                   + 0.1 * torch.randn((case["M"], 2), generator=g, device=DEV)).contiguous()
        st["index"] = ivhd.KnnIndex(X)
    elif kind == "train":
        n = case["batch"] * case["batches"]
        st["X"], lab = _rows("u8", n, case["n_in"], seed, 2)
        g = _gen(seed, 4)
        T = torch.randn((20, 2), generator=g, device=DEV)[lab] \
            + 0.1 * torch.randn((n, 2), generator=g, device=DEV)
        st["T"] = ((T - T.mean(0)) / T.std(0)).contiguous()
        st["p0"] = _net_params(case["n_in"], case["hidden"], seed)
        st["net"] = ivhd.MLP(case["n_in"], case["hidden"], max_batch=case["batch"])
    elif kind == "place":
        if case["dtype"] == "u8":
            st["X"], _ = _rows("u8", case["n"], case["n_in"], seed, 2)
            st["scale"] = 1 / 255
        else:
            X = torch.rand((case["n"], case["n_in"]), generator=_gen(seed, 2), device=DEV)
            st["X"] = X.to(torch.bfloat16) if case["dtype"] == "bf16" else X
            st["scale"] = 1.0
        st["net"] = ivhd.MLP(case["n_in"], case["hidden"], max_batch=65536)
        st["net"].set_params(_net_params(case["n_in"], case["hidden"], seed))
    else:
        g = _gen(seed)
        st["knn"], lab = _graph(case["M"], case["k"], g)
        centre = 10 * torch.rand((50, 2), generator=g, device=DEV)
        st["Y"] = (centre[lab] + 0.3 * torch.randn((case["M"], 2), generator=g, device=DEV)).contiguous()
        st["labels"] = lab.to(torch.int32)
        st["rows"] = torch.randperm(case["M"], generator=g, device=DEV)[:case["rows"]].sort().values
    return st


# ---- one pass -------------------------------------------------------------------


def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "embed":
        with ivhd.Embedding(st["knn"], r=case["r"], c=0.01, opt=case["opt"], a=0.9, b=case["b"],
                            pos_format=case["pos"], seed=st["seed"]) as emb:
            if not case["report"]:
                emb.step(case["steps"])
                return {"positions": emb.positions()}
            curve = []
            for s in range(0, case["steps"], case["report"]):
                emb.step(min(case["report"], case["steps"] - s))
                curve.append(emb.stress())
            return {"positions": emb.positions(), "stress": np.array(curve)}
    if kind == "batch":
        with ivhd.Embedding.batch(st["graphs"], [r for _, _, r in st["shapes"]], st["seed"],
                                  c=0.01, a=0.9, b=0.001) as emb:
            emb.step(case["steps"])
            return {"positions": emb.positions()}
    if kind == "knn":
        return {"knn": ivhd.knn_build(st["X"], case["k"])}
    if kind == "query":
        ids = st["index"].query(st["Q"], case["k"])
        return {"ids": ids, "placed": ivhd.place_nn(st["Y"], ids)}
    if kind == "train":
        net, B = st["net"], case["batch"]
        net.set_params(st["p0"])
        for s in range(case["batches"]):
            loss = net.train_step(st["X"][s * B:(s + 1) * B], st["T"][s * B:(s + 1) * B], lr=1e-3,
                                  x_scale=1 / 255, want_loss=s == case["batches"] - 1)
        return {"params": net.get_params(), "loss": loss}
    if kind == "place":
        return {"y": st["net"].forward(st["X"], x_scale=st["scale"])}
    q, low = ivhd.eval_qnx(st["Y"], st["knn"], st["rows"], return_lowd=True)
    return {"qnx": q, "neighbours": low,
            "cf": ivhd.eval_cf(st["Y"], st["labels"], case["nn"], st["rows"])}


# ---- what a pass cannot do without ------------------------------------------------


def _embed_work(M, k, r, steps, half):
    # each step reads and writes every position and velocity once (and the half-precision copy)
    # and reads each term once from both of its endpoints' rows; each term is about 12
    # operations for its two endpoints and each update 8
    terms = M * (k + r)
    return (steps * (32.0 * M + (8.0 * M if half else 0) + 8.0 * terms) + 4.0 * M * k + 8.0 * M,
            steps * (24.0 * terms + 8.0 * M))


def work(case):
    kind = case["kind"]
    if kind == "embed":
        b, f = _embed_work(case["M"], case["k"], case["r"], case["steps"], case["pos"] != "f32")
        if case["opt"] == "adadelta":
            b += 16.0 * case["M"] * case["steps"]
        return {"bytes": b, "flops": f}
    if kind == "batch":
        w = [_embed_work(M, k, r, case["steps"], False) for M, k, r in _batch_shapes(case, 64)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    if kind == "knn":
        e = 1 if case["dtype"] == "u8" else 4
        # every unordered pair once, two operations per feature
        return {"bytes": case["M"] * (case["N"] * e + 4.0 * case["k"]),
                "flops": float(case["M"]) * (case["M"] - 1) * case["N"]}
    if kind == "query":
        e = 1 if case["dtype"] == "u8" else 4
        return {"bytes": (case["M"] + case["Mq"]) * float(case["N"] * e) + case["Mq"] * (4.0 * case["k"] + 8),
                "flops": 2.0 * case["M"] * case["Mq"] * case["N"]}
    H, n_in = case.get("hidden", 0), case.get("n_in", 0)
    params = H * n_in + H * H + 4 * H + 2
    if kind == "train":
        n = case["batch"] * case["batches"]
        # forward and the two backward products (no input gradient), weights and moments per step
        return {"bytes": n * (n_in + 8.0) + case["batches"] * 24.0 * params,
                "flops": n * (4.0 * H * n_in + 6.0 * H * H + 12.0 * H)}
    if kind == "place":
        e = {"u8": 1, "bf16": 2, "f32": 4}[case["dtype"]]
        return {"bytes": case["n"] * (n_in * e + 8.0) + 4.0 * params,
                "flops": case["n"] * (2.0 * H * n_in + 2.0 * H * H + 4.0 * H)}
    # two criteria, one squared distance (5 operations) per row and point
    return {"bytes": case["M"] * (8.0 + 4.0 * case["k"] + 4) + case["rows"] * (8.0 + 4.0 * case["k"]),
            "flops": 5.0 * case["M"] * case["rows"]}


def tolerance(case):
    """About four times what was measured against 64 bits (embeddings in 32 bits) or against the
    same 16-bit roundings with every sum taken in 64 bits (the network)."""
    kind = case["kind"]
    if kind in ("embed", "batch"):
        if case.get("opt") == "adadelta":
            return {"rel": 2e-3, "max": 0.14}  # 4.4e-4, 0.034: each step divides by the gradient's size
        if case.get("pos") == "f16":
            return {"rel": 6e-4, "max": 0.04}  # 1.4e-4, 0.008
        if case.get("pos") == "bf16":
            return {"rel": 8e-3, "max": 0.04}  # 2e-3, 0.01
        return {"rel": 2e-5, "max": 0.02}  # 6e-6
    if kind == "train":
        return {"rel": 3e-3, "max": 0.3}  # weights after some tens of Adam steps, each divided by its gradient's size
    if kind == "place":
        return {"rel": 1e-3, "max": 0.025}  # 2.4e-4, 0.0053
    return "exact"  # ids, counts and the positions they select


# ---- the same in 64 bits ------------------------------------------------------------


def _s64(v):
    v &= (1 << 64) - 1
    return v - (1 << 64) if v >> 63 else v


_GAMMA, _MUL1, _MUL2 = _s64(0x9E3779B97F4A7C15), _s64(0xBF58476D1CE4E5B9), _s64(0x94D049BB133111EB)


def _shr(z, n):
    return (z >> n) & ((1 << (64 - n)) - 1)


def _sm64(seed, t):
    """Output t of SplitMix64 seeded with seed (int64 tensors, arithmetic modulo 2^64)."""
    z = seed + (t + 1) * _GAMMA
    z = (z ^ _shr(z, 30)) * _MUL1
    z = (z ^ _shr(z, 27)) * _MUL2
    return z ^ _shr(z, 31)


def _streams(M, seed, domain):
    key = torch.full((M,), _s64(int(seed) ^ domain), dtype=torch.int64, device=DEV)
    return _sm64(key, torch.arange(M, device=DEV))


def _random_neighbours(knn, r, seed):
    M = knn.shape[0]
    s = _streams(M, seed, 0x726E5F6C69737473)
    out = torch.full((M, r), -1, dtype=torch.int64, device=DEV)
    got = torch.zeros(M, dtype=torch.int64, device=DEV)
    todo = torch.arange(M, device=DEV)
    for t in range(64 * r):
        x = _sm64(s[todo], torch.full_like(todo, t))
        j = _shr(_shr(x, 32) * M + _shr((x & 0xFFFFFFFF) * M, 32), 32)
        ok = (j != todo) & ~(knn[todo] == j[:, None]).any(1) & ~(knn[j] == todo[:, None]).any(1) \
            & ~(out[todo] == j[:, None]).any(1)
        i = todo[ok]
        out[i, got[i]] = j[ok]
        got[i] += 1
        todo = todo[got[todo] < r]
        if todo.numel() == 0:
            return out
    raise RuntimeError("a vertex without enough eligible random neighbours")


def _stress64(y, a, b, ra, rb, c):
    dn = (y[a] - y[b]).square().sum(1)
    d = (y[ra] - y[rb]).square().sum(1).sqrt()
    return float(dn.sum() + c * (1 - d).square().sum())


def _embed64(knn, r, seed, steps, opt, b, report=0, c=0.01, a=0.9, rho=0.95, eps=1e-6):
    M, k = knn.shape
    knn = knn.long()
    rn = _random_neighbours(knn, r, seed)
    s = _streams(M, seed, 0x696E69745F706F73)
    zero = torch.zeros_like(s)
    y = torch.stack([_shr(_sm64(s, zero + q), 40) for q in (0, 1)], 1).double() * 2.0 ** -24
    own = torch.arange(M, device=DEV)
    na, nb = own.repeat_interleave(k), knn.reshape(-1)
    ra, rb = own.repeat_interleave(r), rn.reshape(-1)
    # the attraction is linear: a sparse matrix with the neighbour counts on its diagonal
    i = torch.cat([na, nb])
    j = torch.cat([nb, na])
    adj = torch.sparse_coo_tensor(torch.stack([i, j]), torch.ones(i.numel(), dtype=torch.float64, device=DEV),
                                  (M, M)).coalesce().to_sparse_csr()
    deg = torch.bincount(i, minlength=M).double()[:, None]
    v, e2 = torch.zeros_like(y), torch.zeros_like(y)

    def force(p):
        f = adj @ p - deg * p
        u = p[rb] - p[ra]
        d = u.square().sum(1, keepdim=True).sqrt()
        g = torch.where(d > 0, c * (1 - 1 / d), torch.zeros_like(d)) * u
        f.index_add_(0, ra, g)
        f.index_add_(0, rb, g, alpha=-1)
        return f

    curve = []
    for n in range(steps):
        if opt == "adadelta":
            g = -force(y)
            v = rho * v + (1 - rho) * g * g
            dx = -((e2 + eps).sqrt() / (v + eps).sqrt()) * g
            e2 = rho * e2 + (1 - rho) * dx * dx
            y = y + dx
        else:
            f = force(y + a * v if opt == "nesterov" else y)
            v = a * v + b * f
            y = y + v
        if report and ((n + 1) % report == 0 or n + 1 == steps):
            curve.append(_stress64(y, na, nb, ra, rb, c))
    return y, curve


def _net64(flat, n_in, H):
    p, at = [], 0
    for shape in ((H, n_in), (H,), (H, H), (H,), (2, H), (2,)):
        n = math.prod(shape)
        p.append(flat[at:at + n].double().reshape(shape))
        at += n
    return p


def _gelu64(z):
    return 0.5 * z * (1 + torch.erf(z * math.sqrt(0.5)))


def _gelu_grad64(z):
    return 0.5 * (1 + torch.erf(z * math.sqrt(0.5))) + z * torch.exp(-0.5 * z * z) / math.sqrt(2 * math.pi)


def _train64(st):
    case, B = st["case"], st["case"]["batch"]
    p = _net64(st["p0"], case["n_in"], case["hidden"])
    m, v = [torch.zeros_like(q) for q in p], [torch.zeros_like(q) for q in p]
    for s in range(case["batches"]):
        x = st["X"][s * B:(s + 1) * B].double() / 255
        t = st["T"][s * B:(s + 1) * B].double()
        z1 = x @ p[0].T + p[1]
        h1 = _gelu64(z1)
        z2 = h1 @ p[2].T + p[3]
        h2 = _gelu64(z2)
        dy = h2 @ p[4].T + p[5] - t
        loss = float(dy.square().sum() / B)
        dy = 2 * dy / B
        d2 = (dy @ p[4]) * _gelu_grad64(z2)
        d1 = (d2 @ p[2]) * _gelu_grad64(z1)
        g = [d1.T @ x, d1.sum(0), d2.T @ h1, d2.sum(0), dy.T @ h2, dy.sum(0)]
        c1, c2 = 1 - 0.9 ** (s + 1), 1 - 0.999 ** (s + 1)
        for q in range(6):
            m[q] = 0.9 * m[q] + 0.1 * g[q]
            v[q] = 0.999 * v[q] + 0.001 * g[q] * g[q]
            p[q] = p[q] - 1e-3 * (m[q] / c1) / ((v[q] / c2).sqrt() + 1e-8)
    return {"params": torch.cat([q.reshape(-1) for q in p]).cpu().numpy(), "loss": loss}


def exact(case, seed):
    kind = case["kind"]
    if kind == "knn" or (kind == "query" and case["dtype"] != "u8"):
        return None  # ids; near ties of float rows are decided in 32 bits by definition
    st = prepare(case, seed)
    if kind == "embed":
        if case["M"] * (case["k"] + case["r"]) * case["steps"] > 2e10:
            return None
        y, curve = _embed64(st["knn"], case["r"], seed, case["steps"], case["opt"], case["b"],
                            case["report"])
        return {"positions": y, "stress": np.array(curve)} if case["report"] else {"positions": y}
    if kind == "batch":
        return {"positions": torch.cat([
            _embed64(g, r, int(seed) + e, case["steps"], "momentum", 0.001)[0]
            for e, (g, (_, _, r)) in enumerate(zip(st["graphs"], st["shapes"]))])}
    if kind == "query":
        X, Q = st["X"].double(), st["Q"].double()
        n = X.square().sum(1)
        placed = []
        for s in range(0, case["Mq"], 2048):
            d = n[None, :] - 2 * (Q[s:s + 2048] @ X.T)
            # ties go to the lower id: distances and ids are integers, so one key holds both
            key = (d - d.min()) * case["M"] + torch.arange(case["M"], device=DEV)
            ids = key.topk(case["k"], dim=1, largest=False).indices
            placed.append(st["Y"].double()[ids].mean(1))
        return {"ids": None, "placed": torch.cat(placed)}
    if kind == "train":
        return _train64(st)
    if kind == "place":
        p = _net64(_net_params(case["n_in"], case["hidden"], seed), case["n_in"], case["hidden"])
        y = []
        for s in range(0, case["n"], 65536):
            x = st["X"][s:s + 65536].double() * st["scale"]
            h = _gelu64(_gelu64(x @ p[0].T + p[1]) @ p[2].T + p[3])
            y.append(h @ p[4].T + p[5])
        return {"y": torch.cat(y)}
    # neighbours in 64 bits, of which the criteria are counts
    Y, rows, lab = st["Y"].double(), st["rows"], st["labels"]
    hit, same = 0, 0
    n = max(case["k"], case["nn"])
    for s in range(0, rows.numel(), 512):
        r = rows[s:s + 512]
        d = (Y[r, None, 0] - Y[None, :, 0]).square() + (Y[r, None, 1] - Y[None, :, 1]).square()
        d[torch.arange(r.numel(), device=DEV), r] = math.inf
        near = d.topk(n, dim=1, largest=False).indices
        hit += int((near[:, :case["k"], None] == st["knn"][r].long()[:, None, :]).any(2).sum())
        same += int((lab[near[:, :case["nn"]]] == lab[r][:, None]).sum())
    return {"qnx": hit / (case["k"] * rows.numel()), "neighbours": None,
            "cf": same / (case["nn"] * rows.numel())}
