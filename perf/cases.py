"""What the library is timed on: whole calls of its public entry points, over the sizes its users run.

Indexes are IVF-PQ indexes of seeded synthetic vectors with the shapes of this repository's workloads
(Gaussian mixture, SIFT-, Deep-, GIST- and embedding-shaped), built here with plain torch and handed to
``Index``. A program builds an index once and searches it with many batches, so an index depends on its
shape alone and is kept; ``seed`` makes the queries (or the vectors to train on).
"""
import math

import numpy as np
import torch

import paper_2606_07156_gb300 as amp

DEV = "cuda:0"
KSUB = 256

# ---------------------------------------------------------------- the cases

_A = dict(data="gauss", n=20_000, dim=128, nlist=64, M=16)
_SIFT = dict(data="sift", n=1_000_000, dim=128, nlist=1024, M=32)
_DEEP = dict(data="deep", n=10_000_000, dim=96, nlist=4096, M=48)
_GIST = dict(data="gist", n=1_000_000, dim=960, nlist=1024, M=120)
_EMB = dict(data="embed", n=1_000_000, dim=768, nlist=2048, M=96)


def listed():
    return [
        # one request on a small index: the latency of a call
        dict(_A, name="single_small", call="search", nq=1, nprobe=8, k=10, mode="plain", cl="fp32"),
        # odd sizes throughout: a dimension that is no multiple of 16, padded sub-spaces, 12-bit tables
        dict(name="ragged_12bit", call="search", data="gauss", n=50_021, dim=100, nlist=333, M=20, nq=777, nprobe=19,
             k=37, mode="fixed", bits=12, cl="fp32"),
        # online serving of a large index: a few requests at a time, the call captured as a graph
        dict(_DEEP, name="online_deep", call="graph", nq=16, nprobe=32, k=10, mode="mlp", cl="fp32"),
        # batches on a 1M index: full-precision tables, and 8-bit tables with more probes
        dict(_SIFT, name="sift_plain", call="search", nq=10_000, nprobe=32, k=10, mode="plain", cl="fp32"),
        dict(_SIFT, name="sift_8bit", call="search", nq=10_000, nprobe=64, k=10, mode="fixed", bits=8, cl="fp32"),
        # the benchmark's batch on 10M vectors: full precision, and the learned widths with the FP16 coarse stage
        dict(_DEEP, name="deep_plain", call="search", nq=10_000, nprobe=32, k=10, mode="plain", cl="fp32"),
        dict(_DEEP, name="deep_learned", call="search", nq=10_000, nprobe=32, k=10, mode="mlp", cl="fp16"),
        # uneven batch from host buffers: Zipf list sizes, Zipf nprobe, k of 1, 10 or 100 a query
        dict(_GIST, name="gist_uneven_host", call="host", nq=4096, nprobe=128, k=100, mode="fixed", bits=8, cl="fp32",
             uneven=True),
        # embeddings: many sub-spaces, short lists, k = 100, the two-pass search the autotuner picks there
        dict(_EMB, name="embed_k100", call="search", nq=4096, nprobe=64, k=100, mode="fixed", bits=8, cl="fp16",
             kernel="split"),
        # the coarse stage alone at the largest number of lists
        dict(name="locate_fp16", call="locate", data="embed", n=65_536, dim=768, nlist=8192, M=96, nq=20_000, nprobe=64,
             cl="fp16"),
        # offline: labels and training of the precision predictor (forward, backward, Adam)
        dict(_SIFT, name="predictor", call="predictor", nq=2000, nprobe=32, k=10, epochs=2),
        # offline: index training and encoding
        dict(name="train_index", call="train", data="deep", n=200_000, dim=96, nlist=256, M=48, iters=10),
    ]


def draw(rng):
    logu = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    call = rng.choice(["search"] * 6 + ["graph", "host", "locate"])
    data = rng.choice(["gauss", "sift", "deep", "gist", "embed"])
    dim, Ms = rng.choice([(48, (12, 24)), (96, (24, 48)), (100, (20, 50)), (128, (16, 32)), (136, (17, 34)), (200, (25, 40)),
                          (256, (32, 64)), (384, (48, 96)), (768, (96,)), (960, (120,))])
    n = logu(5_000, 1_000_000)
    nlist = max(16, n // logu(120, 2500))
    case = dict(call=call, data=data, n=n + rng.randrange(97), dim=dim, nlist=nlist, M=rng.choice(Ms),
                nq=logu(1, 10_000), nprobe=rng.randint(1, min(64, nlist)), cl=rng.choice(["fp32", "fp32", "fp16", "bf16"]))
    if call == "locate":
        return case
    case["k"] = rng.choice([1, 5, 10, 10, 20, 32, 50, 100, 128])
    case["mode"] = rng.choice(["plain", "plain", "fixed", "fixed", "mlp"])
    if case["mode"] == "fixed":
        case["bits"] = rng.choice([4, 6, 8, 8, 12, 16])
    if rng.random() < 0.2:
        case["uneven"] = True
    # no more than the largest listed case: table entries and look-ups of the probed lists
    cost = case["nprobe"] * case["M"] * (n / nlist + 4 * KSUB)
    case["nq"] = max(1, min(case["nq"], int(3.0e10 / cost)))
    return case


# ---------------------------------------------------------------- data

_SEEDS = {"gauss": 1, "sift": 2, "deep": 3, "gist": 4, "embed": 5}
_COMP = {"gauss": 64, "sift": 1024, "deep": 4096, "gist": 1024, "embed": 8192}


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


class _Mixture:
    """The distribution of one data set: a mixture, its parameters fixed by the data set's own seed."""

    def __init__(self, data, dim, n):
        g = _gen(1000 * _SEEDS[data] + dim)
        k = self.k = max(16, min(_COMP[data], n // 60))
        self.data, self.dim = data, dim
        self.p = torch.ones(k, device=DEV)
        if data == "gauss":
            self.mu = torch.rand(k, dim, generator=g, device=DEV) * 2 - 1
            self.sig = torch.rand(k, 1, generator=g, device=DEV) * 0.25 + 0.05
        elif data == "sift":
            self.w = torch.rand(k, dim, generator=g, device=DEV) * 1.75 + 0.25
        elif data == "deep":
            self.mu = torch.randn(k, dim, generator=g, device=DEV) / math.sqrt(dim)
            self.sig = torch.rand(k, 1, generator=g, device=DEV) * 0.15 + 0.05
            self.rot = torch.linalg.qr(torch.randn(32, dim, dim, generator=g, device=DEV))[0]
            self.decay = torch.arange(1, dim + 1, device=DEV).float().rsqrt()
        elif data == "gist":
            self.p = 1.0 / torch.arange(1, k + 1, device=DEV).float()
            self.scale = 1.0 / (torch.rand(k, dim, generator=g, device=DEV) * 3.5 + 0.5)
        else:
            mu = torch.randn(k, dim, generator=g, device=DEV)
            self.mu = mu / mu.norm(dim=1, keepdim=True)
            self.kappa = torch.rand(k, 1, generator=g, device=DEV) * 180 + 20

    def sample(self, n, g):
        step = 1 << 18
        return torch.cat([self._sample(min(step, n - s), g) for s in range(0, n, step)])

    def _sample(self, n, g):
        d = self.dim
        c = torch.multinomial(self.p, n, replacement=True, generator=g)
        z = torch.randn(n, d, generator=g, device=DEV)
        if self.data == "gauss":
            return self.mu[c] + self.sig[c] * z
        if self.data == "sift":
            return (z.square_().mul_(20.0 * self.w[c])).round_().clamp_(0, 255)  # Gamma(1/2, 40 w)
        if self.data == "deep":
            z *= self.sig[c] * self.decay
            x = torch.empty_like(z)
            for r in range(self.rot.shape[0]):
                i = torch.nonzero(c % self.rot.shape[0] == r)[:, 0]
                x[i] = self.mu[c[i]] + z[i] @ self.rot[r].T
            return x / x.norm(dim=1, keepdim=True)
        if self.data == "gist":
            u = torch.rand(n, d, generator=g, device=DEV).clamp_(1e-7, 1.0)
            return u.log_().neg_().mul_(self.scale[c])
        # von Mises-Fisher, near its mean resultant length (kappa is well below the dimension)
        w = (self.kappa[c] / (d - 1)).clamp(max=0.95) + torch.randn(n, 1, generator=g, device=DEV) / math.sqrt(d)
        w = w.clamp(-0.99, 0.99)
        v = z - (z * self.mu[c]).sum(1, keepdim=True) * self.mu[c]
        return w * self.mu[c] + (1 - w * w).sqrt() * (v / v.norm(dim=1, keepdim=True))


def _nearest(X, C, chunk=1 << 16):
    cn = (C * C).sum(1)
    return torch.cat([(cn - 2.0 * (x @ C.T)).argmin(1) for x in X.split(chunk)])


def _kmeans(X, k, iters):
    """Lloyd iterations from evenly spaced rows (sums by matrix products: the same on every run)."""
    C = X[torch.arange(k, device=DEV) * X.shape[0] // k].clone()
    for _ in range(iters):
        a = _nearest(X, C)
        sums, cnt = torch.zeros_like(C), torch.zeros(k, 1, device=DEV)
        for x, b in zip(X.split(1 << 16), a.split(1 << 16)):
            hot = (b[None, :] == torch.arange(k, device=DEV)[:, None]).float()
            sums += hot @ x
            cnt += hot.sum(1, keepdim=True)
        C = torch.where(cnt > 0, sums / cnt.clamp_min(1), C)
    return C


_kept = {}


def _keep(key, make, most=48):
    if key not in _kept:
        while len(_kept) >= most:
            _kept.pop(next(iter(_kept)))
        _kept[key] = make()
    return _kept[key]


def _geometry(case):
    return tuple(case[f] for f in ("data", "n", "dim", "nlist", "M"))


def _mixture(case):
    return _keep(("mixture", case["data"], case["dim"], case["n"]), lambda: _Mixture(case["data"], case["dim"], case["n"]))


def _arrays(case):
    """centroids [nlist, D], codebooks [M, 256, D/M], codes [n, M], list_of [n] of the case's index (torch, GPU)."""
    def make():
        n, dim, nlist, M = (case[f] for f in ("n", "dim", "nlist", "M"))
        X = _mixture(case).sample(n, _gen(77))
        sample = X[torch.arange(min(n, 32 * nlist), device=DEV) * n // min(n, 32 * nlist)]
        C = _kmeans(sample, nlist, 4)
        lo = _nearest(X, C)
        s = torch.arange(min(n, 16384), device=DEV) * n // min(n, 16384)
        R = (X[s] - C[lo[s]]).reshape(len(s), M, dim // M).transpose(0, 1).contiguous()
        B = R[:, torch.arange(KSUB, device=DEV) * len(s) // KSUB].contiguous()
        for _ in range(4):
            a = (B.square().sum(2)[:, None, :] - 2.0 * torch.bmm(R, B.transpose(1, 2))).argmin(2)
            for m in range(M):
                hot = (a[m][None, :] == torch.arange(KSUB, device=DEV)[:, None]).float()
                cnt = hot.sum(1, keepdim=True)
                B[m] = torch.where(cnt > 0, (hot @ R[m]) / cnt.clamp_min(1), B[m])
        yn = B.square().sum(2)[:, None, :]
        codes = torch.empty(n, M, dtype=torch.uint8, device=DEV)
        for i in range(0, n, 1 << 15):
            r = (X[i:i + (1 << 15)] - C[lo[i:i + (1 << 15)]]).reshape(-1, M, dim // M).transpose(0, 1)
            codes[i:i + (1 << 15)] = (yn - 2.0 * torch.bmm(r, B.transpose(1, 2))).argmin(2).T.to(torch.uint8)
        return tuple(t.cpu().numpy() for t in (C, B, codes, lo.to(torch.int32)))
    return _keep(("arrays",) + _geometry(case), make)


def _index(case):
    def make():
        index = amp.Index(*_arrays(case))
        index.set_kernel(case.get("kernel", "auto"))
        index.set_predictor(_predictor(0.0))
        return index
    return _keep(("index", case.get("kernel", "auto")) + _geometry(case), make)


def _predictor(jitter):
    """Weights of a precision predictor: 4 bits for the far probes, wider tables for the near ones (or, with
    ``jitter``, initial weights to train from)."""
    r = np.random.RandomState(9)
    p = dict(W1=np.zeros((32, 5)), b1=np.zeros(32), W2=np.zeros((32, 32)), b2=np.zeros(32), W3=np.zeros((5, 32)), b3=np.zeros(5),
             mean=np.zeros(5), inv_std=np.ones(5))
    if jitter:
        p.update(W1=r.uniform(-jitter, jitter, (32, 5)), W2=r.uniform(-jitter / 2, jitter / 2, (32, 32)),
                 W3=r.uniform(-jitter / 2, jitter / 2, (5, 32)))
        p["inv_std"] = np.array([0.02, 0.005, 0.005, 0.03, 3.0])
    else:
        p["W1"][0, 4], p["W1"][1, 0], p["W2"][0, 0], p["W2"][0, 1] = 1.0, 0.05, 1.0, 1.0
        p["W3"][0, 0], p["W3"][4, 0] = 16.0, -16.0
        p["b3"][:] = [-1.0, -8.0, 0.0, -8.0, 0.5]
    return {f: np.asarray(v, np.float32) for f, v in p.items()}


# ---------------------------------------------------------------- a pass


def _queries(case, seed):
    return _mixture(case).sample(case["nq"], _gen(10_000 + int(seed)))


def _per_query(case, seed):
    """nprobe (Zipf) and k (1, 10 or the largest) of each query of an uneven batch, int32."""
    if not case.get("uneven"):
        return None, None
    r = np.random.RandomState(int(seed) % (1 << 31))
    v = np.arange(1, case["nprobe"] + 1)
    w = v ** -1.1
    ks = [min(x, case["k"]) for x in (1, 10, case["k"])]
    return r.choice(v, case["nq"], p=w / w.sum()).astype(np.int32), r.choice(ks, case["nq"]).astype(np.int32)


def _policy(case):
    if case["mode"] == "mlp":
        return amp.policy("mlp", width_map=True, cl=case["cl"])
    return amp.policy(case["mode"], bits=case.get("bits", 8), cl=case["cl"])


def prepare(case, seed):
    call = case["call"]
    if call == "train":
        return dict(case=case, base=_mixture(case).sample(case["n"], _gen(10_000 + int(seed))))
    state = dict(graph=None, case=case, index=_index(case), q=_queries(case, seed))
    if call == "locate":
        return state
    if call == "predictor":
        classes = np.full(256, 255, np.uint8)
        classes[[4, 6, 8, 12, 16, 0]] = [0, 1, 2, 3, 4, 4]
        state.update(classes=torch.from_numpy(classes).to(DEV), weights=_predictor(1.0),
                     cfg=amp.train_cfg(epochs=case["epochs"], seed=int(seed) % 1000))
        return state
    pq, kq = _per_query(case, seed)
    state["pol"] = _policy(case)
    if call == "host":
        state["q"] = state["q"].cpu().pin_memory()
        out = (torch.empty(case["nq"], case["k"], dtype=torch.int64).pin_memory(),
               torch.empty(case["nq"], case["k"], dtype=torch.float32).pin_memory())
        state.update(pq=pq, kq=kq, out=out)
        return state
    state.update(pq=None if pq is None else torch.from_numpy(pq).to(DEV), kq=None if kq is None else torch.from_numpy(kq).to(DEV))
    if call == "graph":
        state["graph"], *state["out"] = state["index"].capture_graph(state["q"], case["nprobe"], case["k"], state["pol"],
                                                                     state["pq"], state["kq"])
    return state


def run(state):
    case, call = state["case"], state["case"]["call"]
    if call == "train":
        index = amp.Index.train(state["base"], case["nlist"], case["M"], iters=case["iters"], pq_iters=case["iters"])
        arrays = index.export()
        index.close()
        return arrays
    index = state["index"]
    if call == "locate":
        return index.locate(state["q"], case["nprobe"], case["cl"])
    if call == "predictor":
        feat, labels = index.make_training_set(state["q"], case["nprobe"], case["k"])
        cls = state["classes"][labels.long()]
        return dict(features=feat, labels=labels, weights=index.mlp_train(state["weights"], feat, cls, state["cfg"]))
    if call == "graph":
        state["graph"].launch()
        return tuple(state["out"])
    if call == "host":
        return index.search_host(state["q"], case["nprobe"], case["k"], state["pol"], state["pq"], state["kq"], out=state["out"])
    return index.search(state["q"], case["nprobe"], case["k"], state["pol"], state["pq"], state["kq"])


# ---------------------------------------------------------------- what a pass cannot do without


def work(case):
    n, dim, nlist, M = (case[f] for f in ("n", "dim", "nlist", "M"))
    index = nlist * dim * 4 + KSUB * dim * 4
    if case["call"] == "train":
        sample = min(n, 256 * nlist)
        flops = 2.0 * dim * (sample * nlist * case["iters"] + 65_536 * KSUB * case["iters"] + n * nlist + n * KSUB)
        return dict(bytes=n * dim * 4 + index + n * (M + 8), flops=flops)
    nq, nprobe = case["nq"], case["nprobe"]
    locate = 2.0 * nq * nlist * dim
    if case["call"] == "locate":
        return dict(bytes=nq * dim * 4 + nlist * dim * 4 + nq * nprobe * 8, flops=locate)
    mean_probe = nprobe if not case.get("uneven") else float((np.arange(1, nprobe + 1) ** -0.1).sum() / (np.arange(1, nprobe + 1) ** -1.1).sum())
    pairs = nq * mean_probe
    touched = nlist * (1.0 - (1.0 - mean_probe / nlist) ** nq)  # lists probed by any query
    tables = 2.0 * nq * KSUB * dim + pairs * M * KSUB
    flops = locate + tables + pairs * (n / nlist) * M
    out = nq * nprobe * 21 if case["call"] == "predictor" else nq * case["k"] * 12
    return dict(bytes=nq * dim * 4 + index + touched * (n / nlist) * M + out, flops=flops)


# ---------------------------------------------------------------- in 64 bits


def exact(case, seed):
    """The distances in 64 bits (searches with one table width, the coarse stage, the predictor's features)."""
    call = case["call"]
    if call == "train" or case.get("mode") == "mlp" or case["n"] > 10_000_000:
        return None
    C, B, codes, lo = (torch.from_numpy(a).to(DEV) for a in _arrays(case))
    C, B = C.double(), B.double()
    nq, nprobe, M, dim = case["nq"], case["nprobe"], case["M"], case["dim"]
    q = _queries(case, seed).double()
    D2, P = [], []
    for x in q.split(2048):
        d = torch.stack([((x - c) ** 2).sum(1) for c in C], 1) if len(C) <= 64 else \
            ((x * x).sum(1)[:, None] + (C * C).sum(1) - 2.0 * (x @ C.T)).clamp_min_(0)
        v, i = d.topk(nprobe, dim=1, largest=False)
        D2.append(v)
        P.append(i)
    D2, P = torch.cat(D2), torch.cat(P)
    if call == "locate":
        return None, D2.float()
    order = torch.argsort(lo, stable=True)
    ends = torch.cumsum(torch.bincount(lo, minlength=case["nlist"]), 0).cpu().tolist()
    bits = case.get("bits", 8) if case.get("mode") == "fixed" else 0
    k = case["k"]
    pq, kq = _per_query(case, seed)
    rank = torch.arange(nprobe, device=DEV)
    use = torch.ones(nq, nprobe, dtype=torch.bool, device=DEV) if pq is None else rank[None, :] < torch.from_numpy(pq).to(DEV)[:, None]
    if call == "predictor":
        radius = torch.zeros(case["nlist"], dtype=torch.float64, device=DEV)
        yn = (B * B).sum(2)
        norm2 = yn[torch.arange(M, device=DEV), codes.long()].sum(1)
        radius = radius.scatter_reduce(0, lo.long(), norm2, "amax").sqrt()
        size = torch.bincount(lo, minlength=case["nlist"]).double()
        D = D2.sqrt()
        j = (rank.double() / nprobe).expand(nq, nprobe)
        feat = torch.stack([D - D[:, :1], radius[P[:, :1]].expand(nq, nprobe), radius[P], size[P].sqrt(), j], 2)
        return dict(features=feat, labels=None, weights=None)
    best = torch.full((nq, nprobe, k), math.inf, dtype=torch.float64, device=DEV)
    mm = torch.arange(M, device=DEV)
    for l, end in enumerate(ends):
        begin = ends[l - 1] if l else 0
        qi, ji = torch.nonzero((P == l) & use, as_tuple=True)
        if not len(qi) or begin == end:
            continue
        code = codes[order[begin:end]].long()
        for s in range(0, len(qi), 512):
            a, j = qi[s:s + 512], ji[s:s + 512]
            if not bits:
                x = (C[l] + B[mm, code].reshape(len(code), dim))
                y = q[a]
                d = (y - C[l]).square().sum(1)[:, None] + (x - C[l]).square().sum(1) - 2.0 * ((y - C[l]) @ (x - C[l]).T)
            else:
                r = (q[a] - C[l]).reshape(len(a), M, dim // M)
                T = (B * B).sum(2) - 2.0 * torch.einsum("qmj,mcj->qmc", r, B)
                lowest = T.amin(2, keepdim=True)
                span = (T - lowest).amax((1, 2))
                top = 2.0 ** bits - 1
                t = torch.round((T - lowest) * torch.where(span > 0, top / span, 0.0)[:, None, None]).float()
                S = torch.zeros(len(a), len(code), device=DEV)
                for m in range(M):
                    S += t[:, m].index_select(1, code[:, m])
                d = (r * r).sum((1, 2))[:, None] + lowest.sum((1, 2))[:, None] + S.double() * (span / top)[:, None]
            w = min(k, d.shape[1])
            best[a, j, :w] = d.topk(w, dim=1, largest=False, sorted=False)[0]
    d = best.reshape(nq, -1).topk(k, dim=1, largest=False)[0]
    if kq is not None:
        d = torch.where(torch.arange(k, device=DEV)[None, :] < torch.from_numpy(kq).to(DEV)[:, None], d, math.inf)
    return None, d
