"""Performance cases: the calls a user of the library makes, over the sizes it is used at.

A program loads a graph once (``Graph``), sets its options, and then asks for
single-source scores (``query``), top-k lists (``topk``), batches of sources
(``*_batch``), or runs the steps of a query on its own buffers (``forward``,
``allocate``, ``reverse``, top-k selection).  Every case prepares the graph and the
buffers and times one such call.  Graphs are the seeded recipes of ``synth`` drawn on
the GPU: Erdos-Renyi, Chung-Lu with Pareto weights, R-MAT.  The server's waves run the
batch calls' launch sequence, so the batch cases stand for it.
"""
import math

import numpy as np
import torch

import paper_2004_03493_gb300 as esim

KAPPA = 4.0  # the walk budget the benchmark and the exceed-rate test use; 0 is the paper's constant


def listed():
    return [
        # an interactive lookup on a small graph: the smallest call, launches and latency
        dict(name="topk_er2k", kind="topk", graph="er", n=2000, m=20000, c=0.6, eps=1e-2, kappa=KAPPA, k=50),
        # the paper's own sample constant (Theorem 1's guarantee): walk pairs alone
        dict(name="query_er2k_guarantee", kind="query", graph="er", n=2000, m=20000, c=0.6, eps=1e-3, kappa=0.0),
        # Algorithm 3 as the paper gives it: every node explores to its own depth
        dict(name="query_er3k_paper_depth", kind="query", graph="er", n=3001, m=30011, c=0.6, eps=1e-3, kappa=KAPPA,
             alg3=1, alg3_rule=0),
        # the benchmark's query: power-law graph, eps 1e-6, top-50, cost-model depths
        dict(name="topk_cl100k", kind="topk", graph="cl", n=100000, m=1000000, gamma=2.1, c=0.6, eps=1e-6, kappa=KAPPA,
             k=50, alg3=1, alg3_rule=1, alg3_max_depth=8, alg3_max_nodes=128, alg3_overlap=5),
        # a score vector brought to the host, with the library's default cost-model options
        dict(name="query_cl20k_host", kind="query_host", graph="cl", n=20011, m=200003, gamma=2.1, c=0.6, eps=1e-5,
             kappa=KAPPA, alg3=1, alg3_rule=1),
        # the precision form end to end at a moderate eps (Algorithm 2)
        dict(name="topk_cl100k_fp32c", kind="topk", graph="cl", n=100003, m=1000003, gamma=2.1, c=0.6, eps=1e-3,
             kappa=KAPPA, k=100, precision=1),
        # sparse linearization on a million nodes: FP64 sweeps, kept entries only
        dict(name="query_cl1m_sparse", kind="query", graph="cl", n=1000003, m=17500001, gamma=2.2, c=0.6, eps=1e-3,
             kappa=KAPPA, sparse_hist=1),
        # a full batch: 64 sources, each with its own eps, top-100
        dict(name="batch_topk_rmat17_64", kind="topk_batch", graph="rmat", n=1 << 17, m=3750000, c=0.6, eps=5e-5,
             eps_hi=1e-3, kappa=KAPPA, B=64, k=100),
        # a small wave of requests: 5 sources, whole score vectors
        dict(name="batch_query_cl20k_5", kind="query_batch", graph="cl", n=20011, m=200003, gamma=2.1, c=0.6, eps=1e-3,
             eps_hi=1e-2, kappa=KAPPA, B=5),
        # the sweeps at L = 33 (eps 1e-7) on a million nodes: forward, allocation, reverse; FP64 and FP32c
        dict(name="sweeps_cl1m_fp64", kind="sweeps", graph="cl", n=1000003, m=17500001, gamma=2.2, c=0.6, eps=1e-7,
             kappa=KAPPA, precision=0),
        dict(name="sweeps_cl1m_fp32c", kind="sweeps", graph="cl", n=1000003, m=17500001, gamma=2.2, c=0.6, eps=1e-7,
             kappa=KAPPA, precision=1),
        # top-k selection over a program's own scores
        dict(name="select_1m", kind="select", n=1048573, k=100),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case: the kinds above with sizes, densities, eps and options over their ranges."""
    kind = rng.choice(["topk", "query", "paper", "cost", "cost", "precision", "sparse", "batch", "batch", "sweeps",
                       "sweeps", "select"])
    c = rng.choice([0.6, 0.6, 0.6, 0.5, 0.7])
    if kind == "select":
        return dict(kind="select", n=int(_log(rng, 1000, 4e6)) | 1, k=int(_log(rng, 1, 4096)))
    if kind in ("topk", "query"):
        n = int(_log(rng, 500, 20000))
        m = int(n * rng.uniform(3, 20)) | 1
        d = dict(kind=kind, graph="er", n=n, m=m, c=c, eps=_log(rng, 1e-3, 1e-2),
                 kappa=rng.choice([KAPPA, KAPPA, 0.0]))
        if kind == "topk":
            d["k"] = int(_log(rng, 1, 400))
        return d
    if kind == "paper":
        n = int(_log(rng, 500, 3000))
        return dict(kind="query", graph="er", n=n, m=int(n * rng.uniform(5, 12)) | 1, c=0.6, eps=_log(rng, 1e-3, 1e-2),
                    kappa=KAPPA, alg3=1, alg3_rule=0)
    if kind == "batch":
        scale = rng.randint(11, 17)
        d = dict(kind=rng.choice(["topk_batch", "query_batch"]), graph="rmat", n=1 << scale,
                 m=int((1 << scale) * rng.uniform(4, 28)) | 1, c=c, eps=_log(rng, 1e-4, 1e-3), eps_hi=1e-2, kappa=KAPPA,
                 B=rng.randint(1, 64))
        if d["kind"] == "topk_batch":
            d["k"] = int(_log(rng, 1, 400))
        return d
    if kind == "cost":
        n = int(_log(rng, 5000, 100000))
        d = dict(kind=rng.choice(["topk", "query_host"]), graph="cl", n=n, m=int(n * rng.uniform(5, 10)) | 1, gamma=2.1,
                 c=0.6, eps=_log(rng, 1e-6, 1e-4), kappa=KAPPA, alg3=1, alg3_rule=1)
        if d["kind"] == "topk":
            d["k"] = int(_log(rng, 1, 400))
        return d
    n = int(_log(rng, 2000, 1e6))
    m = int(n * rng.uniform(4, 17.5)) | 1
    d = dict(graph="cl", n=n, m=m, gamma=rng.choice([2.1, 2.2, 2.5]), c=c, kappa=KAPPA)
    if kind == "precision":
        return dict(d, kind="topk", eps=_log(rng, 1e-3, 1e-2), k=int(_log(rng, 1, 400)), precision=1)
    if kind == "sparse":
        return dict(d, kind="query", eps=_log(rng, 1e-3, 1e-2), sparse_hist=1)
    return dict(d, kind="sweeps", eps=_log(rng, 1e-7, 1e-3), precision=rng.choice([0, 1]))


# ---------------------------------------------------------------- inputs


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _graph(case, seed):
    """(rowptr int64, col int32) on the device: row j lists the in-neighbours of node j."""
    dev = _device()
    n, m = case["n"], case["m"]
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed * 7919 + 17)

    def rand(k):
        return torch.rand(k, generator=gen, device=dev, dtype=torch.float64)

    if case["graph"] == "cl":
        w = 1.0 / (case["gamma"] - 1.0)
        cdfs = []
        for _ in range(2):
            t = torch.cumsum((1.0 - rand(n)) ** (-w), 0)
            cdfs.append(t / t[-1])

        def endpoints(k):
            return [torch.searchsorted(t, rand(k), right=True).clamp_(max=n - 1) for t in cdfs]
    elif case["graph"] == "rmat":
        perm = torch.randperm(n, generator=gen, device=dev)

        def endpoints(k):
            s = torch.zeros(k, dtype=torch.int64, device=dev)
            d = torch.zeros(k, dtype=torch.int64, device=dev)
            for _ in range(n.bit_length() - 1):
                r = rand(k)
                q = (r >= 0.57).long() + (r >= 0.76).long() + (r >= 0.95).long()
                s = (s << 1) | (q >> 1)
                d = (d << 1) | (q & 1)
            return perm[s], perm[d]
    else:
        def endpoints(k):
            return [torch.randint(0, n, (k,), generator=gen, device=dev) for _ in range(2)]

    keys = torch.empty(0, dtype=torch.int64, device=dev)
    count = int(m * 1.3) + 256
    for _ in range(12):
        s, d = endpoints(count)
        keep = s != d
        keys = torch.unique(torch.cat([keys, d[keep] * n + s[keep]]))
        if keys.numel() >= m:
            break
        count = 2 * (m - keys.numel()) + int(0.3 * m)
    if keys.numel() > m:
        keys = keys[torch.randperm(keys.numel(), generator=gen, device=dev)[:m]].sort().values
    dst = keys // n
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    rowptr[1:] = torch.cumsum(torch.bincount(dst, minlength=n), 0)
    return rowptr, (keys - dst * n).to(torch.int32)


def _sources(rowptr, count, seed):
    """Uniform sources among the nodes with an in-edge."""
    din = (rowptr[1:] - rowptr[:-1]).cpu().numpy()
    return np.random.default_rng(seed).choice(np.flatnonzero(din > 0), size=count, replace=True).astype(np.int64)


def _batch_eps(case, seed):
    lo, hi = math.log(case["eps"]), math.log(max(case["eps"], case["eps_hi"]))
    return np.exp(np.random.default_rng(seed + 1).uniform(lo, hi, case["B"]))


def _scores(case, seed):
    """SimRank-like scores: a few large, a long tail, exact zeros and ties."""
    gen = torch.Generator(device=_device())
    gen.manual_seed(seed)
    n = case["n"]
    t = torch.rand(n, generator=gen, device=_device(), dtype=torch.float64)
    s = 0.6 * torch.exp(-16.0 * t)
    s[torch.rand(n, generator=gen, device=_device()) < 0.3] = 0.0
    ties = torch.randint(0, n, (max(1, n // 50),), generator=gen, device=_device())
    s[ties] = torch.round(s[ties], decimals=2)
    return s


def _levels(c, eps):
    return int(math.ceil(math.log(2.0 / eps) / math.log(1.0 / c)))


def _dhat(case, seed):
    """A diagonal in the range of D: uniform in [1 - c, 1]."""
    gen = torch.Generator(device=_device())
    gen.manual_seed(seed + 5)
    return (1.0 - case["c"]) + case["c"] * torch.rand(case["n"], generator=gen, device=_device(), dtype=torch.float64)


OPTIONS = ("kappa", "precision", "sparse_hist", "alg3", "alg3_rule", "alg3_max_depth", "alg3_max_nodes", "alg3_overlap")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "select":
        k = min(case["k"], case["n"])
        return dict(case=case, k=k, scores=_scores(case, seed), exclude=seed % case["n"],
                    ids=torch.empty(k, dtype=torch.int32, device="cuda"),
                    vals=torch.empty(k, dtype=torch.float64, device="cuda"))
    rowptr, col = _graph(case, seed)
    n = case["n"]
    g = esim.Graph(n, rowptr.cpu().numpy(), col.cpu().numpy(), **{o: case[o] for o in OPTIONS if o in case})
    st = dict(case=case, g=g, seed=seed, u=_sources(rowptr, case.get("B", 1), seed))
    if kind == "topk":
        st["ids"] = torch.empty(case["k"], dtype=torch.int32, device="cuda")
        st["vals"] = torch.empty(case["k"], dtype=torch.float64, device="cuda")
    elif kind == "query":
        st["s"] = torch.empty(n, dtype=torch.float64, device="cuda")
    elif kind in ("topk_batch", "query_batch"):
        st["eps"] = _batch_eps(case, seed)
        if kind == "topk_batch":
            st["ids"] = torch.empty((case["B"], case["k"]), dtype=torch.int32, device="cuda")
            st["vals"] = torch.empty((case["B"], case["k"]), dtype=torch.float64, device="cuda")
        else:
            st["s"] = torch.empty((case["B"], n), dtype=torch.float64, device="cuda")
    elif kind == "sweeps":
        L = _levels(case["c"], case["eps"])
        st.update(L=L, R_b=esim.esim_sample_base(n, case["c"], case["eps"], case["kappa"]), dhat=_dhat(case, seed),
                  hist=torch.empty((L + 1) * n, dtype=torch.float32 if case["precision"] else torch.float64,
                                   device="cuda"),
                  pi=torch.empty(n, dtype=torch.float64, device="cuda"),
                  R=torch.empty(n, dtype=torch.uint64, device="cuda"),
                  off=torch.empty(n + 1, dtype=torch.uint64, device="cuda"),
                  s=torch.empty(n, dtype=torch.float64, device="cuda"))
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "select":
        esim.esim_select_topk_static(st["scores"], case["n"], st["exclude"], st["k"], st["ids"], st["vals"],
                                     torch.cuda.current_stream())
        return st["ids"], st["vals"]
    g, c = st["g"], case["c"]
    if kind == "topk":
        return g.topk_device(int(st["u"][0]), c, case["eps"], case["k"], st["seed"], st["ids"], st["vals"])
    if kind == "query":
        return g.query_device(int(st["u"][0]), c, case["eps"], st["seed"], st["s"])
    if kind == "query_host":
        return g.query(int(st["u"][0]), c, case["eps"], st["seed"])
    if kind == "topk_batch":
        return g.topk_batch_device(st["u"], st["eps"], c, case["k"], st["seed"], st["ids"], st["vals"])
    if kind == "query_batch":
        return g.query_batch_device(st["u"], st["eps"], c, st["seed"], st["s"])
    u, L = int(st["u"][0]), st["L"]
    if case["precision"]:
        g.forward_f32(u, c, L, st["hist"])
        g.allocate_f32(st["hist"], L, st["R_b"], 0, st["pi"], st["R"], st["off"])
        g.reverse_f32(st["hist"], L, c, st["dhat"], st["s"])
    else:
        g.forward(u, c, L, st["hist"])
        g.allocate(st["hist"], L, st["R_b"], 0, st["pi"], st["R"], st["off"])
        g.reverse(st["hist"], L, c, st["dhat"], st["s"])
    # R(k) of this eps is a count up to 1e13 decided by the last bits of pi: pi itself is returned
    return st["hist"], st["pi"], st["s"]


# ---------------------------------------------------------------- what a pass cannot do without


def _pairs(case, eps):
    """Walk pairs of one Algorithm 2 query: R_b ||pi||^2, the source's own (1 - sqrt c)^2 and a tenth more."""
    a = 1.0 - math.sqrt(case["c"])
    kappa = case["kappa"] if case["kappa"] > 0 else 6.0 / a ** 4
    return kappa * math.log(case["n"]) / (eps * eps) * a * a * 1.1


def work(case):
    if case["kind"] == "select":
        return {"bytes": 8 * case["n"] + 12 * case["k"], "flops": case["n"]}
    n, m, c = case["n"], case["m"], case["c"]
    B = case.get("B", 1)
    eps = [case["eps"]] if B == 1 else list(_batch_eps(case, 0))
    value = 4 if case.get("precision") or "batch" in case["kind"] else 8
    csr = 4 * m + 4 * (n + 1)
    L = max(_levels(c, e / 2 if case.get("sparse_hist") else e) for e in eps)
    # per level: both CSRs once; x, pi^l and the next x; s, pi^l, D^ and the next s, per column
    nbytes = L * (2 * csr + B * n * (3 * value + 8 + 8 + 8 + value)) + 8 * B * n
    flops = 4.0 * m * L * B
    if case["kind"] != "sweeps" and not case.get("alg3"):
        # 48 integer operations a pair-step (a Philox-4x32-10 block and the step), 1/(1-c) steps a pair
        flops += sum(_pairs(case, e / 2 if case.get("sparse_hist") else e) for e in eps) * 48.0 / (1.0 - c)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits, plain torch

_M32 = 0xFFFFFFFF


def _philox(x0, x1, x2, x3, seed):
    """Philox-4x32-10 (Salmon et al., SC'11) on int64 tensors that hold 32-bit words."""
    k0, k1 = seed & _M32, (seed >> 32) & _M32
    for _ in range(10):
        p0, p1 = x0 * 0xD2511F53, x2 * 0xCD9E8D57  # 64-bit products; the sign bit is data
        x0, x1, x2, x3 = (((p1 >> 32) & _M32) ^ x1 ^ k0, p1 & _M32, ((p0 >> 32) & _M32) ^ x3 ^ k1, p0 & _M32)
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return x0, x1, x2, x3


def _redraw(rlo, rhi, k, t, walk, d, seed):
    """Lemire's rejection: the first word of the walk's side stream that is not rejected."""
    limit = (2 ** 32 - d) % d
    one = lambda v: torch.tensor([v], dtype=torch.int64)  # noqa: E731
    for j in range(1 << 14):
        for w in _philox(one(rlo), one(rhi), one(k), one(0x80000000 | walk << 30 | j << 16 | t), seed):
            p = int(w) * d
            if (p & _M32) >= limit:
                return p >> 32
    return p >> 32


def _nonmeet(rowptr, col, R, c, seed):
    """How many of the R(k) pairs of sqrt(c)-walks of each node never meet."""
    dev, n = rowptr.device, R.numel()
    first, din, col = rowptr[:-1], rowptr[1:] - rowptr[:-1], col.long()
    T = min(int(math.floor(math.sqrt(c) * 2 ** 32)), _M32)
    off = torch.cumsum(R, 0)
    total = int(off[-1])
    count = torch.zeros(n, dtype=torch.int64, device=dev)
    for g0 in range(0, total, 1 << 23):
        gi = torch.arange(g0, min(total, g0 + (1 << 23)), device=dev)
        k = torch.searchsorted(off, gi, right=True)
        r = gi - (off[k] - R[k])
        a, b = k, k
        t = 0
        while gi.numel():
            w0, w1, w2, w3 = _philox(r & _M32, r >> 32, k, torch.full_like(k, t), seed)
            da, db = din[a], din[b]
            on = (w0 < T) & (w2 < T) & (da > 0) & (db > 0)
            count += torch.bincount(k[~on], minlength=n)
            k, r, gi, a, b, da, db, w1, w3 = (v[on] for v in (k, r, gi, a, b, da, db, w1, w3))
            na, nb = w1 * da, w3 * db
            ia, ib = (na >> 32) & _M32, (nb >> 32) & _M32
            for walk, prod, d, idx in ((0, na, da, ia), (1, nb, db, ib)):
                again = torch.nonzero((prod & _M32) < (2 ** 32 - d) % d.clamp(min=1)).flatten()
                for i in again.tolist():
                    idx[i] = _redraw(int(r[i]) & _M32, int(r[i]) >> 32, int(k[i]), t, walk, int(d[i]), seed)
            a, b = col[first[a] + ia], col[first[b] + ib]
            apart = a != b
            k, r, gi, a, b = (v[apart] for v in (k, r, gi, a, b))
            t += 1
    return count


def _query64(rowptr, col, u, c, eps, kappa, seed, sparse=False):
    n = rowptr.numel() - 1
    if sparse:
        eps = 0.5 * eps
    a = 1.0 - math.sqrt(c)
    kappa = kappa if kappa > 0 else 6.0 / a ** 4
    hist = _forward64(rowptr, col, u, c, _levels(c, eps))
    pi = torch.zeros_like(hist[0])
    for h in hist:
        pi = pi + h
    v = kappa * math.log(n) / (eps * eps) * (pi * pi)
    R = torch.where(pi > 0, torch.ceil(v).clamp(min=1), torch.zeros_like(v)).long()
    D = torch.where(R > 0, _nonmeet(rowptr, col, R, c, seed).double() / R.clamp(min=1).double(), 0.0)
    if sparse:
        hist = [torch.where(h > a * a * eps, h, 0.0) for h in hist]
    return _reverse64(rowptr, col, hist, c, D)


def _rows(rowptr):
    return torch.repeat_interleave(torch.arange(rowptr.numel() - 1, device=rowptr.device), rowptr[1:] - rowptr[:-1])


def _forward64(rowptr, col, u, c, L):
    n, src, dst = rowptr.numel() - 1, col.long(), _rows(rowptr)
    inv = 1.0 / (rowptr[1:] - rowptr[:-1]).clamp(min=1).double()
    h = torch.zeros(n, dtype=torch.float64, device=rowptr.device)
    h[u] = 1.0 - math.sqrt(c)
    hist = [h]
    for _ in range(L):
        hist.append(math.sqrt(c) * torch.zeros_like(h).index_add_(0, src, (hist[-1] * inv)[dst]))
    return hist


def _reverse64(rowptr, col, hist, c, D):
    src, dst = col.long(), _rows(rowptr)
    inv = 1.0 / (rowptr[1:] - rowptr[:-1]).clamp(min=1).double()
    a = 1.0 - math.sqrt(c)
    s = D * hist[-1] / a
    for h in reversed(hist[:-1]):
        s = math.sqrt(c) * inv * torch.zeros_like(s).index_add_(0, dst, s[src]) + D * h / a
    return s


def _top(s, k, exclude):
    """The k largest, (score descending, id ascending), without `exclude`."""
    t = s.clone()
    t[exclude] = -math.inf
    vals, ids = torch.sort(t, descending=True, stable=True)
    k_real = min(k, s.numel() - 1)
    out_i = torch.full((k,), -1, dtype=torch.int32, device=s.device)
    out_v = torch.zeros(k, dtype=torch.float64, device=s.device)
    out_i[:k_real], out_v[:k_real] = ids[:k_real].int(), vals[:k_real]
    return out_i, out_v


def exact(case, seed):
    kind = case["kind"]
    if kind == "select":
        return _top(_scores(case, seed), min(case["k"], case["n"]), seed % case["n"])
    eps = _batch_eps(case, seed) if "B" in case else [case["eps"]]
    pairs = 0 if kind == "sweeps" else sum(_pairs(case, e / 2 if case.get("sparse_hist") else e) for e in eps)
    if case.get("alg3") or pairs > 6e7:  # Lemma 5's terms, or more walks than plain torch takes in seconds
        return None
    rowptr, col = _graph(case, seed)
    c, us = case["c"], _sources(rowptr, case.get("B", 1), seed)
    if kind == "sweeps":
        hist = _forward64(rowptr, col, int(us[0]), c, _levels(c, case["eps"]))
        return torch.cat(hist), torch.stack(hist).sum(0), _reverse64(rowptr, col, hist, c, _dhat(case, seed))
    s = [_query64(rowptr, col, int(u), c, float(e), case["kappa"], seed, bool(case.get("sparse_hist")))
         for u, e in zip(us, eps)]
    if kind in ("topk", "topk_batch"):
        # ids at near-ties are the run's own; the scores have a value
        vals = [_top(v, case["k"], int(u))[1] for v, u in zip(s, us)]
        return None, torch.stack(vals) if "B" in case else vals[0]
    return torch.stack(s) if "B" in case else s[0]
