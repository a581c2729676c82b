"""The work whose speed is measured: calls of the public entry points over the
sizes and options that users of the library have.

Four kinds of case:

``search``  ``Index.search`` (Filter, conditioning, tables, Rank, Select and
            the optional exact rerank) on a loaded index: from one query on
            10^4 rows to 1024-query batches on 10^7 rows, M from 8 to 120
            subspaces, predicates on one, two and three columns, host arrays
            or device tensors.
``encode``  ``ifvs_pq_encode``: the codes of raw vectors under a codebook.
``lloyd``   ``ifvs_pq_train``: the PQ codebook by Lloyd iterations.
``step``    ``ifvs_train_step``: one SGD step of the memory bank, W and w_z
            (mining, loss, gradient, update), with the updated parameters.

Index contents.  Every mixture component has a prototype code (the codeword
nearest to its centre in each subspace); a row keeps each of its component's
codes with probability 1/2 and takes a uniform codeword otherwise.  Queries
are drawn around the components' centres, so a query's neighbours are the
rows of its component that kept most of their codes, at distances that seldom
tie.  Attribute columns: uniform int32, correlated with the component, or a
date and a Zipf-distributed int16 category (and a price).
"""
import ctypes
import math

import numpy as np
import torch

from paper_2607_22922_gb300 import ifvs, synth

DEV = "cuda"
K = 256             # codewords per subspace
H = 2               # hash functions
RANK = 8            # adjustment rank
BANK = 4096         # memory-bank rows
SPAN = {"date": 3650, "uniform": 1_000_000, "price": 10_000}
N_CATEGORIES = 100
SIGMA = 0.3         # spread of a component around its centre
TAU, LAMBDA, LR, LR_WZ = 8.0, 0.001, 5.0, 1e-4   # training step


def listed():
    search = dict(kind="search", ds=8, cond=True, wz=True, rerank=0, host=False)
    return [
        # one query from a program that holds numpy arrays, on a small index:
        # launches, copies and synchronisations
        dict(search, name="one-query-10k-host", n=10_000, m=16, nq=1, k=10, attrs="date", sel=0.1, host=True),
        # one query of an interactive service on 10^6 rows
        dict(search, name="one-query-1m", n=1_000_003, m=16, nq=1, k=10, attrs="date", sel=0.1),
        # a handful of concurrent queries, selective, k = 100, on 10^7 rows
        dict(search, name="few-queries-10m", n=10_000_000, m=16, nq=16, k=100, attrs="uniform", sel=0.01),
        # a full batch whose predicates mix selectivities from 0.1 % to all rows
        dict(search, name="batch-1m-mixed", n=1_000_000, m=16, nq=1024, k=10, attrs="date", sel="mixed"),
        # a full batch of wide windows at k = 100: the largest case
        dict(search, name="batch-10m-wide", n=10_000_000, m=16, nq=1024, k=100, attrs="uniform", sel=0.5),
        # 960-dimensional vectors: M = 120, an attribute correlated with the data
        dict(search, name="batch-m120", n=500_009, m=120, nq=256, k=10, attrs="cluster", sel=0.1),
        # category = c AND a date range on two columns (M = 12)
        dict(search, name="batch-m12-category", n=4_000_037, m=12, nq=512, k=10, attrs="date+category", sel=0.01),
        # category <= c AND a wide date range: the conjunction no sort order covers
        dict(search, name="batch-m12-conjunction", n=4_000_037, m=12, nq=256, k=10, attrs="date+category", sel=0.4),
        # clauses on three columns, plain PQ tables, exact rerank of 100 candidates
        dict(search, name="rerank-3-columns", n=300_007, m=32, nq=100, k=20, attrs="date+category+price", sel=0.02,
             cond=False, wz=False, rerank=100),
        # encoding a slice of a dataset
        dict(kind="encode", name="encode-1m", n=1 << 20, m=16, ds=8, dmin=False),
        # codebook training on the usual sample
        dict(kind="lloyd", name="lloyd-64k", n=65_536, m=16, ds=8, iters=10),
        # one mini-batch of training the memory bank and W on 10^6 rows
        dict(kind="step", name="train-step-1m", n=1_000_000, m=16, ds=8, nq=1024, n_pos=10, n_neg=32, sel=0.1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["search", "encode", "lloyd", "step"], [10, 3, 1, 2])[0]
    if kind == "encode":
        m, ds = rng.choice([(16, 8), (16, 8), (12, 8), (120, 8), (32, 4), (8, 16)])
        n = min(_log(rng, 1000, 1 << 20), (1 << 24) // m)
        return dict(kind=kind, n=n, m=m, ds=ds, dmin=rng.random() < 0.3)
    if kind == "lloyd":
        m, ds = rng.choice([(16, 8), (16, 8), (12, 8), (32, 4)])
        return dict(kind=kind, n=_log(rng, 4096, 1 << 18), m=m, ds=ds, iters=rng.randint(2, 10))
    if kind == "step":
        return dict(kind=kind, n=_log(rng, 20_000, 1_000_000), m=rng.choice([16, 16, 12]), ds=8,
                    nq=_log(rng, 32, 1024), n_pos=rng.randint(1, 10), n_neg=rng.randint(8, 48),
                    sel=rng.choice([0.01, 0.1, 0.5]))
    m, ds = rng.choice([(16, 8)] * 6 + [(12, 8)] * 2 + [(120, 8), (120, 8), (8, 16), (32, 4), (32, 8), (24, 8)])
    attrs = rng.choice(["date", "date", "uniform", "uniform", "cluster", "date+category", "date+category",
                        "date+category+price"])
    n = _log(rng, 10_000, 10_000_000 if m <= 16 else 1_000_000)
    nq = _log(rng, 1, 1024)
    sel = rng.choice([0.001, 0.01, 0.02, 0.1, 0.1, 0.4, 0.5, 1.0, "mixed"])
    if attrs in ("date+category", "date+category+price") and sel in (1.0, "mixed"):
        sel = 0.05
    cost = n * m * (sel if sel != "mixed" else 0.3)
    while nq > 1 and nq * cost > (4e10 if m <= 16 and "+" not in attrs else 1e10):
        nq //= 2
    k = _log(rng, 1, 128)
    rerank = 0
    if n * m * ds <= 10 ** 8 and rng.random() < 0.25:
        rerank = min(256, 2 * k + rng.randint(0, 50))
    cond = rng.random() < 0.75
    return dict(kind=kind, n=n, m=m, ds=ds, nq=nq, k=k, attrs=attrs, sel=sel, cond=cond, wz=rng.random() < 0.75,
                rerank=rerank, host=rng.random() < 0.25)


# ------------------------------------------------------------------ inputs

class State:
    """What a program has in hand before the call."""


def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 1_000_003 + salt)
    return g


def _mixture(case, seed):
    """Centres [clusters][D], codebook [m][K][ds], prototype codes [clusters][m]."""
    m, ds = case["m"], case["ds"]
    g = _gen(seed, 1)
    clusters = max(32, min(1024, case["n"] // 4000))
    centres = torch.randn((clusters, m * ds), generator=g, device=DEV)
    owner = torch.randint(0, clusters, (m, K), generator=g, device=DEV)
    sub = centres.view(clusters, m, ds)
    cb = torch.empty((m, K, ds), device=DEV)
    proto = torch.empty((clusters, m), dtype=torch.uint8, device=DEV)
    for i in range(m):
        cb[i] = sub[owner[i], i] + SIGMA * torch.randn((K, ds), generator=g, device=DEV)
        proto[:, i] = torch.cdist(sub[:, i], cb[i]).argmin(1).to(torch.uint8)
    return centres, cb, proto


def _codes(case, seed, proto, cluster):
    n, m = case["n"], case["m"]
    codes = torch.empty((n, m), dtype=torch.uint8, device=DEV)
    g = _gen(seed, 2)
    step = max(1, (1 << 27) // m)
    for a in range(0, n, step):
        c = proto[cluster[a:a + step]]
        r = torch.randint(0, 1 << 16, c.shape, generator=g, device=DEV, dtype=torch.int32)
        codes[a:a + step] = torch.where(r >= 1 << 15, c, (r & 255).to(torch.uint8))
    return codes


def _attributes(case, seed, cluster, clusters):
    """The columns, as [(name, tensor)]."""
    n, g, cols = case["n"], _gen(seed, 3), []
    for name in case.get("attrs", "date").split("+"):
        if name == "category":
            p = torch.from_numpy(synth.zipf_probs(N_CATEGORIES, 1.1)).to(DEV).cumsum(0)
            a = torch.searchsorted(p, torch.rand(n, generator=g, device=DEV, dtype=torch.float64))
            cols.append((name, a.clamp(max=N_CATEGORIES - 1).to(torch.int16)))
        elif name == "cluster":
            a = cluster * 10 + torch.randint(0, 10, (n,), generator=g, device=DEV)
            cols.append((name, a.to(torch.int32)))
        else:
            a = torch.randint(0, SPAN[name], (n,), generator=g, device=DEV)
            cols.append((name, a.to(torch.int32)))
    return cols


def _predicates(case, seed, clusters, cl):
    """[nq] predicate records of about the wanted selectivity."""
    nq = case["nq"]
    rng = np.random.default_rng([seed, 4])
    names = case.get("attrs", "date").split("+")
    p = synth.empty_predicates(nq)
    sel = case["sel"]
    per_query = np.full(nq, 0.0 if sel == "mixed" else sel)
    if sel == "mixed":
        per_query = rng.choice([0.001, 0.01, 0.1, 0.5, 1.0], size=nq)

    def window(i, clause, col, span, s):
        width = int(min(span, max(1, round(s * span))))
        lo = int(rng.integers(0, span - width + 1))
        synth.set_clause(p[i], clause, col, synth.OP_RANGE, lo, lo + width)

    zipf = synth.zipf_probs(N_CATEGORIES, 1.1)
    cum = np.cumsum(zipf)
    for i in range(nq):
        s = float(per_query[i])
        p[i]["n_clauses"] = len(names)
        if len(names) == 1:
            if names[0] == "cluster":   # a window around the query's own component
                span = clusters * 10
                width = int(min(span, max(1, round(s * span))))
                lo = int(min(max(0, cl[i] * 10 - rng.integers(0, width)), span - width))
                synth.set_clause(p[i], 0, 0, synth.OP_RANGE, lo, lo + width)
            else:
                window(i, 0, 0, SPAN[names[0]], s)
            continue
        if len(names) == 3:              # the price takes part of the selectivity
            synth.set_clause(p[i], 2, 2, synth.OP_LT, SPAN["price"] // 2)
            s = min(1.0, 2.0 * s)
        if s <= zipf[0] and len(names) == 2:
            ok = np.nonzero(zipf >= s)[0]
            c = int(ok[rng.integers(0, len(ok))])
            synth.set_clause(p[i], 0, 1, synth.OP_EQ, c)
            window(i, 1, 0, SPAN["date"], s / zipf[c])
        else:
            c = int(min(np.searchsorted(cum, max(s, 0.3)), N_CATEGORIES - 1))
            synth.set_clause(p[i], 0, 1, synth.OP_LE, c)
            window(i, 1, 0, SPAN["date"], s / cum[c])
    return p


def _conditioning(case, seed, cb):
    """Bank rows ~ N(0, 1/h) (so alpha ~ N(0, 1)) and W of 5 % of the codewords' spread."""
    m, ds = case["m"], case["ds"]
    g = _gen(seed, 5)
    bank = torch.randn((BANK, m * RANK), generator=g, device=DEV) / math.sqrt(H)
    W = torch.randn((m, RANK, K, ds), generator=g, device=DEV) * (0.05 * cb.reshape(m, -1).std(1))[:, None, None, None]
    seeds = np.random.default_rng([seed, 6]).integers(0, 2 ** 63, size=H, dtype=np.int64).astype(np.uint64)
    return bank.cpu().numpy(), W.cpu().numpy(), seeds


def _raw(case, seed):
    """Raw vectors [n][D] of a Gaussian mixture, and K of them as start codewords [m][K][ds]."""
    n, m, ds = case["n"], case["m"], case["ds"]
    g = _gen(seed, 7)
    clusters = 256
    centres = torch.randn((clusters, m * ds), generator=g, device=DEV)
    cl = torch.randint(0, clusters, (n,), generator=g, device=DEV)
    X = centres[cl] + SIGMA * torch.randn((n, m * ds), generator=g, device=DEV)
    rows = torch.randint(0, clusters, (K,), generator=g, device=DEV)
    cb = centres[rows] + SIGMA * torch.randn((K, m * ds), generator=g, device=DEV)
    return X, cb.view(K, m, ds).transpose(0, 1).contiguous()


def _searchable(case, seed):
    """The index's inputs and the queries, shared by prepare and exact."""
    s = State()
    centres, s.cb, proto = _mixture(case, seed)
    clusters = len(centres)
    s.cluster = torch.randint(0, clusters, (case["n"],), generator=_gen(seed, 8), device=DEV)
    s.codes = _codes(case, seed, proto, s.cluster)
    s.cols = _attributes(case, seed, s.cluster, clusters)
    g = _gen(seed, 9)
    cl = torch.randint(0, clusters, (case["nq"],), generator=g, device=DEV)
    s.q = centres[cl] + SIGMA * torch.randn((case["nq"], case["m"] * case["ds"]), generator=g, device=DEV)
    s.query_cluster = cl
    s.preds = _predicates(case, seed, clusters, cl.cpu().numpy())
    s.wz = synth.WZ_IDENTITY + 0.2 * torch.randn(s.q.shape, generator=g, device=DEV)
    s.bank = s.W = s.seeds = None
    if case.get("cond", True):
        s.bank, s.W, s.seeds = _conditioning(case, seed, s.cb)
    s.vectors = None
    if case.get("rerank"):
        noise = 0.5 * SIGMA * torch.randn((case["n"], case["m"] * case["ds"]), generator=g, device=DEV)
        s.vectors = torch.empty_like(noise)
        for i in range(case["m"]):
            a = slice(i * case["ds"], (i + 1) * case["ds"])
            s.vectors[:, a] = s.cb[i][s.codes[:, i].long()] + noise[:, a]
    return s


def _positives(case, seed, s):
    """[nq][n_pos] rows of the query's component inside its window (-1 where there is none)."""
    span = SPAN["date"]
    key, order = (s.cluster * span + s.cols[0][1].long()).sort()
    lo = torch.from_numpy(s.preds["c"][:, 0]["lo"].copy()).to(DEV)
    hi = torch.from_numpy(s.preds["c"][:, 0]["hi"].copy()).to(DEV)
    a = torch.searchsorted(key, s.query_cluster * span + lo)
    b = torch.searchsorted(key, s.query_cluster * span + hi)
    u = torch.rand((case["nq"], case["n_pos"]), generator=_gen(seed, 10), device=DEV, dtype=torch.float64)
    at = a[:, None] + (u * (b - a)[:, None]).long()
    rows = order[at.clamp(max=len(order) - 1)]
    return torch.where((b > a)[:, None], rows, torch.full_like(rows, -1))


def prepare(case, seed):
    if case["kind"] in ("encode", "lloyd"):
        s = State()
        s.case = case
        s.X, s.cb = _raw(case, seed)
        if case["kind"] == "encode":
            s.codes = torch.empty((case["n"], case["m"]), dtype=torch.uint8, device=DEV)
            s.dmin = torch.empty((case["n"], case["m"]), device=DEV) if case["dmin"] else None
        else:
            s.out = torch.empty_like(s.cb)
            s.objective = torch.empty((case["iters"], case["m"]), dtype=torch.float64, device=DEV)
        return s
    t = _searchable(case, seed)
    s = State()
    s.case = case
    s.index = ifvs.Index(t.codes, [c for _, c in t.cols], vectors=t.vectors, D=case["m"] * case["ds"], K=K,
                         device_io=True)
    s.index.load_codebooks(t.cb.cpu().numpy(), bank=t.bank, W=t.W, hash_seeds=t.seeds)
    s.preds, s.q = t.preds, t.q
    s.wz = t.wz if case.get("wz", True) else None
    nq = case["nq"]
    if case["kind"] == "step":
        s.preds = torch.from_numpy(s.preds.view(np.uint8).reshape(nq, -1).copy()).to(DEV)
        s.wz = torch.full((case["m"] * case["ds"],), synth.WZ_IDENTITY, device=DEV)
        s.positives = _positives(case, seed, t)
        s.negatives = torch.empty((nq, case["n_neg"]), dtype=torch.int64, device=DEV)
        s.bank = torch.empty(t.bank.shape, device=DEV)
        s.W = torch.empty(t.W.shape, device=DEV)
    elif case["host"]:
        s.q = s.q.cpu().numpy()
        s.wz = None if s.wz is None else s.wz.cpu().numpy()
    else:
        s.preds = torch.from_numpy(s.preds.view(np.uint8).reshape(nq, -1).copy()).to(DEV)
        s.ids = torch.empty((nq, case["k"]), dtype=torch.int64, device=DEV)
        s.dists = torch.empty((nq, case["k"]), device=DEV)
        s.npass = torch.empty(nq, dtype=torch.int64, device=DEV)
    return s


# -------------------------------------------------------------------- pass

def run(s):
    case = s.case
    if case["kind"] == "encode":
        ifvs.ifvs_pq_encode(s.X, s.cb, codes=s.codes, dmin=s.dmin, flags=ifvs.IFVS_F_DEVICE_IO)
        return {"codes": s.codes, "dmin": s.dmin}
    if case["kind"] == "lloyd":
        ifvs.ifvs_pq_train(s.X, s.cb, case["iters"], C_out=s.out, objective=s.objective, flags=ifvs.IFVS_F_DEVICE_IO)
        return {"codebook": s.out, "objective": s.objective}
    if case["kind"] == "step":
        loss, neg = s.index.train_step(s.q, s.preds, s.wz, s.positives, case["n_neg"], TAU, LAMBDA, LR,
                                       flags=ifvs.IFVS_F_DEVICE_IO, negatives=s.negatives, lr_wz=LR_WZ)
        # the updated parameters, read on the device through the C entry point
        rc = ifvs.lib().ifvs_get_conditioning(s.index.h, ctypes.c_void_p(s.bank.data_ptr()),
                                              ctypes.c_void_p(s.W.data_ptr()), ifvs.IFVS_F_DEVICE_IO)
        if rc != ifvs.IFVS_OK:
            raise RuntimeError(ifvs.ifvs_last_error())
        return {"loss": loss, "negatives": neg, "wz": s.wz, "bank": s.bank, "W": s.W}
    flags = 0 if case["cond"] else ifvs.IFVS_F_PLAIN_PQ
    if case["host"]:
        ids, dists, npass = s.index.search(s.q, s.preds, case["k"], wz=s.wz, rerank=case["rerank"], flags=flags)
    else:
        ids, dists, npass = s.index.search(s.q, s.preds, case["k"], wz=s.wz, rerank=case["rerank"],
                                           flags=flags | ifvs.IFVS_F_DEVICE_IO, ids=s.ids, dists=s.dists,
                                           npass=s.npass)
    return {"ids": ids, "dists": dists, "npass": npass}


def _selectivity(case):
    return 0.322 if case["sel"] == "mixed" else case["sel"]


def work(case):
    n, m, ds = case["n"], case["m"], case["ds"]
    D = m * ds
    if case["kind"] == "encode":
        return {"bytes": 4 * n * D + n * m + 4 * K * D + (4 * n * m if case["dmin"] else 0), "flops": 3 * n * K * D}
    if case["kind"] == "lloyd":
        # each iteration reads the vectors once; the squared differences and the member sums
        return {"bytes": case["iters"] * 4 * n * D + 8 * K * D, "flops": case["iters"] * (3 * n * K * D + n * D)}
    nq, sel = case["nq"], _selectivity(case)
    pool = sel * n
    seen = min(n, nq * pool)             # rows that some query looks at
    attr_bytes = sum(2 if a == "category" else 4 for a in case.get("attrs", "date").split("+"))
    by = seen * m + nq * (8 * D + 104) + 4 * K * D
    fl = nq * pool * m + nq * K * D * 4  # one addition per code; the weighted tables
    if "+" in case.get("attrs", "date"):
        by += n * attr_bytes
    if case.get("cond", True):
        by += 4 * RANK * K * D + nq * H * m * RANK * 4
        fl += nq * 2 * RANK * K * D
    if case["kind"] == "step":
        v = case["n_pos"] + case["n_neg"]
        by += 8 * nq * v + 2 * 4 * (BANK * m * RANK + RANK * K * D)   # candidates, updated bank and W
        fl += nq * v * D * (4 * RANK + 8)
        return {"bytes": by, "flops": fl}
    by += nq * (12 * case["k"] + 8)
    if case["rerank"]:
        by += 4 * nq * case["rerank"] * D
        fl += 3 * nq * case["rerank"] * D
    return {"bytes": by, "flops": fl}


def tolerance(case):
    if case["kind"] == "encode":
        return "exact"                   # the definition fixes the order of every rounding
    if case["kind"] == "lloyd":
        # a mean's last bit can move a row to another codeword: 7e-4 between
        # the argmin in 32 and in 64 bits after ten iterations
        return {"rel": 3e-3, "max": 0.5}
    if case["kind"] == "step":
        # the updated parameters are within 4e-8 of 64 bits
        return {"rel": 1e-6, "max": 4e-5, "differ": 0.002}
    # sums of M float32 entries (5e-8 to 2e-7 from 64 bits); ids differ where
    # two distances meet within them
    return {"rel": 1e-6, "max": 1e-5, "differ": 0.002}


# -------------------------------------------------- the same in 64 bits

def _bank_rows(q, preds, seeds):
    """[nq][h] bank rows of <q, f>: FNV-1a-64 of the key, SplitMix64 finalizer."""
    nq = len(preds)
    qb = np.ascontiguousarray(q, np.float32).view(np.uint8).reshape(nq, -1)
    c = preds["c"]
    clauses = np.concatenate([c["col"][..., None].view(np.uint8).reshape(nq, 4, 4),
                              c["op"][..., None].view(np.uint8).reshape(nq, 4, 4),
                              c["lo"][..., None].view(np.uint8).reshape(nq, 4, 8),
                              c["hi"][..., None].view(np.uint8).reshape(nq, 4, 8)], axis=2).reshape(nq, -1)
    head = np.ascontiguousarray(preds["n_clauses"]).view(np.uint8).reshape(nq, 4)
    key = np.concatenate([qb, head, clauses], axis=1).astype(np.uint64)
    used = qb.shape[1] + 4 + 24 * preds["n_clauses"].astype(np.int64)
    h = np.full(nq, 14695981039346656037, np.uint64)
    with np.errstate(over="ignore"):
        for i in range(key.shape[1]):
            h = np.where(i < used, (h ^ key[:, i]) * np.uint64(1099511628211), h)
        out = []
        for s in seeds:
            z = h ^ s
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xbf58476d1ce4e5b9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94d049bb133111eb)
            out.append((z ^ (z >> np.uint64(31))) % np.uint64(BANK))
    return torch.from_numpy(np.stack(out, 1).astype(np.int64)).to(DEV)


def _tables(case, s, alpha, W, wf):
    """Weighted distance tables [nq][m][K] in 64 bits."""
    m, ds, nq = case["m"], case["ds"], case["nq"]
    q = s.q.double().view(nq, m, ds)
    lut = torch.empty((nq, m, K), dtype=torch.float64, device=DEV)
    for i in range(m):
        c = s.cb[i].double()[None]
        if alpha is not None:
            c = c + (alpha.view(nq, m, RANK)[:, i] @ W[i].reshape(RANK, K * ds)).view(nq, K, ds)
        lut[:, i] = (wf.view(nq, m, 1, ds)[:, i] * (q[:, i, None] - c) ** 2).sum(-1)
    return lut


def _passes(col, p, lo_clause):
    """Rows of one column against one clause of every query: [nq][rows]."""
    op, lo, hi = (torch.from_numpy(np.ascontiguousarray(p["c"][:, lo_clause][f]).astype(np.int64)).to(DEV)[:, None]
                  for f in ("op", "lo", "hi"))
    v = col.long()[None]
    ok = torch.zeros((len(p), len(col)), dtype=torch.bool, device=DEV)
    ok |= (op == synth.OP_EQ) & (v == lo)
    ok |= (op == synth.OP_RANGE) & (v >= lo) & (v < hi)
    ok |= (op == synth.OP_LT) & (v < lo)
    ok |= (op == synth.OP_LE) & (v <= lo)
    return ok


def _best(case, s, lut, k):
    """The k smallest distances of each query's pool, and their rows: [nq][k], inf and -1 where the pool ends."""
    nq, n, m = case["nq"], case["n"], case["m"]
    d = torch.full((nq, k), math.inf, dtype=torch.float64, device=DEV)
    ids = torch.full((nq, k), -1, dtype=torch.int64, device=DEV)
    step = max(1024, min(n, (1 << 26) // nq))
    for a in range(0, n, step):
        b = min(n, a + step)
        codes = s.codes[a:b].long()
        acc = torch.zeros((nq, b - a), dtype=torch.float64, device=DEV)
        for i in range(m):
            acc += lut[:, i].index_select(1, codes[:, i])
        for c in range(int(s.preds["n_clauses"][0])):
            col = int(s.preds["c"][0, c]["col"])
            acc.masked_fill_(~_passes(s.cols[col][1][a:b], s.preds, c), math.inf)
        near, at = acc.topk(min(k, b - a), 1, largest=False)
        both, which = torch.cat([d, near], 1).topk(k, 1, largest=False)
        ids = torch.cat([ids, at + a], 1).gather(1, which)
        d = both
    return d, torch.where(torch.isinf(d), torch.full_like(ids, -1), ids)


def exact(case, seed):
    if case["kind"] in ("encode", "lloyd"):
        X, cb = _raw(case, seed)
        X, cb = X.double(), cb.double()
        n, m, ds = case["n"], case["m"], case["ds"]
        X = X.view(n, m, ds)
        if case["kind"] == "encode":
            if not case["dmin"]:
                return None
            dmin = torch.empty((n, m), dtype=torch.float64, device=DEV)
            for i in range(m):
                for a in range(0, n, 1 << 16):
                    dmin[a:a + (1 << 16), i] = _nearest(X[a:a + (1 << 16), i], cb[i])[0]
            return {"codes": None, "dmin": dmin}
        obj = torch.empty((case["iters"], m), dtype=torch.float64, device=DEV)
        for it in range(case["iters"]):
            for i in range(m):
                parts = [_nearest(X[a:a + (1 << 16), i], cb[i]) for a in range(0, n, 1 << 16)]
                d, code = torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts])
                obj[it, i] = d.sum()
                count = torch.zeros(K, dtype=torch.float64, device=DEV).index_add_(0, code, torch.ones_like(d))
                total = torch.zeros((K, ds), dtype=torch.float64, device=DEV).index_add_(0, code, X[:, i].contiguous())
                cb[i] = torch.where(count[:, None] > 0, total / count.clamp(min=1)[:, None], cb[i])
                for c in (count == 0).nonzero().flatten().tolist():
                    far = int(d.argmax())
                    cb[i, c] = X[far, i]
                    d[far] = 0.0
        return {"codebook": cb, "objective": obj}
    s = _searchable(case, seed)
    nq, m, ds = case["nq"], case["m"], case["ds"]
    rows = alpha = W = None
    if s.bank is not None:
        rows = _bank_rows(s.q.cpu().numpy(), s.preds, s.seeds)
        alpha = torch.from_numpy(s.bank).to(DEV).double()[rows].sum(1)
        W = torch.from_numpy(s.W).to(DEV).double()
    if case["kind"] == "step":
        return _exact_step(case, seed, s, rows, W)
    wf = torch.nn.functional.softplus(s.wz.double()) if case["wz"] else torch.ones_like(s.q, dtype=torch.float64)
    lut = _tables(case, s, alpha, W, wf)
    if not case["rerank"]:
        return {"ids": None, "dists": _best(case, s, lut, case["k"])[0], "npass": None}
    ids = _best(case, s, lut, case["rerank"])[1]
    d = ((s.vectors.double()[ids.clamp(min=0)] - s.q.double()[:, None]) ** 2).sum(-1)
    d = torch.where(ids < 0, torch.full_like(d, math.inf), d)
    return {"ids": None, "dists": d.topk(case["k"], 1, largest=False)[0], "npass": None}


def _nearest(x, c):
    return ((x[:, None] - c[None]) ** 2).sum(-1).min(1)


def _exact_step(case, seed, s, rows, W):
    """The step by automatic differentiation in 64 bits."""
    nq, m, ds, P, Nn = case["nq"], case["m"], case["ds"], case["n_pos"], case["n_neg"]
    pos = _positives(case, seed, s)
    bank = torch.from_numpy(s.bank).to(DEV).double().requires_grad_()
    W = W.clone().requires_grad_()
    wz = torch.full((m * ds,), synth.WZ_IDENTITY, device=DEV).double().requires_grad_()
    alpha = bank[rows].sum(1)
    wf = torch.nn.functional.softplus(wz)
    with torch.no_grad():
        lut = _tables(case, s, alpha, W, wf.expand(nq, -1))
        mined = _best(case, s, lut, P + Nn)[1]
    keep = (mined >= 0) & ~(mined[:, :, None] == pos[:, None, :]).any(-1)
    order = (~keep).to(torch.int8).argsort(dim=1, stable=True)[:, :Nn]
    neg = torch.where(keep.gather(1, order), mined.gather(1, order), torch.full_like(order, -1))
    cand = torch.cat([pos, neg], 1)
    code = s.codes[cand.clamp(min=0)].long()                     # [nq][v][m]
    dist = torch.zeros(cand.shape, dtype=torch.float64, device=DEV)
    anchor = torch.zeros(nq, dtype=torch.float64, device=DEV)
    q = s.q.double().view(nq, m, ds)
    for i in range(m):
        delta = (alpha.view(nq, m, RANK)[:, i] @ W[i].reshape(RANK, K * ds)).view(nq, K, ds)
        anchor = anchor + (delta ** 2).sum((1, 2))
        c = s.cb[i].double()[code[:, :, i]] + delta.gather(1, code[:, :, i, None].expand(-1, -1, ds))
        dist = dist + (wf.view(m, ds)[i] * (q[:, i, None] - c) ** 2).sum(-1)
    logit = torch.where(cand >= 0, -dist / TAU, torch.full_like(dist, -math.inf))
    lp, ln = logit[:, :P], logit[:, P:]
    there = cand[:, :P] >= 0
    safe = torch.where(there, lp, torch.zeros_like(lp))
    each = torch.logsumexp(torch.cat([safe[:, :, None], ln[:, None].expand(-1, P, -1)], 2), 2) - safe
    each = torch.where(there, each, torch.zeros_like(each)).sum(1) / there.sum(1).clamp(min=1)
    loss = (each + LAMBDA * anchor).mean()
    loss.backward()
    with torch.no_grad():
        return {"loss": float(loss), "negatives": None, "wz": wz - LR_WZ * wz.grad, "bank": bank - LR * bank.grad,
                "W": W - LR * W.grad}
