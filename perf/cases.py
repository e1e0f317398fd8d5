"""Performance cases of the SIVF clustering library.

A case is one piece of work that a user's program hands to the library
through its public entry points (the Python binding, or the C ABI it wraps):

  run      cluster a corpus from seeded centroids: sivf_reseed, then sivf_run
           (Algorithm 1) for a few iterations or to convergence;
  resume   continue from saved labels late in a run, when most clusters are
           invariant and the ICP filter acts: sivf_reseed, sivf_set_labels,
           sivf_update, sivf_run;
  update   the update step alone: labels made elsewhere go in, unit centroids
           come out (sivf_set_labels, sivf_update), for two labelings that
           differ in a part of the objects;
  batch    independent corpora in one context (sivf_batch_run);
  build    the allocation-free inverted-file build.

Corpora are seeded Zipf tf-idf documents, made on the GPU with the recipe of
this repository's synthetic corpora: Zipf(s) ranks under a random
permutation, lognormal lengths, distinct terms by rejection of repeats,
tf = 1 + Poisson(1), value = tf ln(N / df), unit rows.
"""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_2103_16141_gb300 import SIVF, SIVFBatch, sivf as S


def listed():
    return [
        # a small corpus clustered to convergence, iterations on the device: launches and latency count
        dict(name="small_run_fp32", kind="run", N=2_000, D=5_000, k=50, s=1.1, mean=39.6, sigma=0.6, precision="fp32",
             icp=1, iters=30, graph=True),
        # a few hundred short texts, the smallest problem a program hands over
        dict(name="tiny_run_bf16", kind="run", N=311, D=1_501, k=13, s=1.1, mean=25.0, sigma=0.6, precision="bf16",
             icp=1, iters=10, graph=False),
        # long documents (about 190 terms), k = 1000: the first iterations from the seeds
        dict(name="medium_run_fp32", kind="run", N=300_000, D=100_000, k=1_000, s=1.05, mean=189.6, sigma=0.7,
             precision="fp32", icp=1, iters=5, graph=False),
        # the same corpus late in its run, continued from saved labels: most objects are filtered
        dict(name="medium_resume_fp32", kind="resume", N=300_000, D=100_000, k=1_000, s=1.05, mean=189.6, sigma=0.7,
             precision="fp32", icp=1, done=30, iters=6, graph=False),
        # ragged sizes, FP16 postings, no filter (Algorithm 2)
        dict(name="ragged_run_fp16", kind="run", N=60_007, D=61_003, k=3_001, s=1.1, mean=120.0, sigma=0.7,
             precision="fp16", icp=0, iters=4, graph=False),
        # 10,000 clusters, BF16 postings
        dict(name="wide_run_bf16", kind="run", N=300_000, D=140_000, k=10_000, s=1.1, mean=91.8, sigma=0.8,
             precision="bf16", icp=1, iters=4, graph=False),
        # 20,000 clusters over short documents: the regime of the 8M-document workload, BF16 postings
        dict(name="large_run_bf16", kind="run", N=500_000, D=140_000, k=20_000, s=1.1, mean=60.0, sigma=0.8,
             precision="bf16", icp=1, iters=4, graph=False),
        # thousands of clusters in the middle of a run, continued from saved labels, iterations on the device
        dict(name="large_resume_bf16", kind="resume", N=400_003, D=140_000, k=8_000, s=1.1, mean=60.0, sigma=0.8,
             precision="bf16", icp=1, done=4, iters=6, graph=True),
        # 20,000 clusters with FP32 postings
        dict(name="large_run_fp32", kind="run", N=100_000, D=140_000, k=20_000, s=1.1, mean=60.0, sigma=0.8,
             precision="fp32", icp=1, iters=4, graph=False),
        # independent corpora of mixed sizes in one context, FP16 postings, iterations on the device
        dict(name="batch_run_fp16", kind="batch", n_inst=16, sizes=3, scale=0.2, precision="fp16", icp=1, iters=20,
             graph=True),
        # new means from given labels, a tenth of the objects changing cluster each time
        dict(name="medium_update_fp32", kind="update", N=300_000, D=100_000, k=1_000, s=1.05, mean=189.6, sigma=0.7,
             precision="fp32", change=0.1),
        # the allocation-free inverted-file build near its size limit
        dict(name="build_noalloc", kind="build", k=1_000, D=100_000, entries=1_000_000),
    ]


def _log_uniform(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def draw(rng: random.Random):
    kind = rng.choice(["run", "run", "run", "resume", "update", "batch", "build"])
    if kind == "build":
        k, D = int(_log_uniform(rng, 8, 50_000)), int(_log_uniform(rng, 1_000, 262_144))
        return dict(kind=kind, k=k, D=D, entries=int(_log_uniform(rng, 2_000, min(1_048_576, k * D / 4))))
    precision = rng.choice(["fp32", "bf16", "fp16"])
    graph = rng.random() < 0.5
    if kind == "batch":
        return dict(kind=kind, n_inst=rng.randint(2, 16), sizes=rng.randint(0, 999), scale=round(_log_uniform(rng, 0.02, 0.2), 4),
                    precision=precision, icp=1, iters=rng.randint(5, 20), graph=graph)
    N = int(_log_uniform(rng, 300, 400_000))
    D = int(_log_uniform(rng, 1_500, 140_000))
    mean = round(_log_uniform(rng, 15.0, min(190.0, D / 20.0)), 1)
    k = int(_log_uniform(rng, 8, max(16, min(20_000, N // 12))))
    case = dict(kind=kind, N=N, D=D, k=k, s=rng.choice([1.05, 1.1]), mean=mean, sigma=rng.choice([0.6, 0.7, 0.8]),
                precision=precision)
    if kind == "update":
        return dict(case, change=round(_log_uniform(rng, 0.01, 0.5), 3))
    # no more work than the largest listed case (500,000 x 20,000 scores of 60 terms, four iterations)
    iters = rng.randint(3, 12)
    cost = N * float(k) * mean
    iters = max(2, min(iters, int(2.0e12 / cost)))
    if kind == "resume":
        return dict(case, icp=1, done=max(3, min(20, int(4.0e12 / cost))), iters=iters, graph=graph)
    return dict(case, icp=rng.choice([1, 1, 1, 0]), iters=iters, graph=graph)


# ---------------------------------------------------------------- inputs

def _corpus(N, D, s, mean, sigma, seed, lo=5, hi=3000):
    """CSR of a Zipf tf-idf corpus on the GPU (int64 row_ptr, int32 idx, float32 val)."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(seed)
    cdf = np.cumsum(np.arange(1, D + 1, dtype=np.float64) ** -s)
    cdf = torch.from_numpy(cdf / cdf[-1]).to(dev)
    term_of = torch.randperm(D, device=dev, generator=g)
    mu = math.log(mean) - sigma * sigma / 2.0
    want = torch.exp(mu + sigma * torch.randn(N, device=dev, generator=g, dtype=torch.float64)).round()
    want = want.clamp(lo, min(hi, D // 4)).to(torch.int64)
    keys = torch.empty(0, dtype=torch.int64, device=dev)
    docs = torch.arange(N, device=dev)
    need = want
    for _ in range(12):  # repeats are drawn again; the few still missing after that are left out
        doc = torch.repeat_interleave(docs, need)
        if doc.numel() == 0:
            break
        r = torch.searchsorted(cdf, torch.rand(doc.numel(), device=dev, generator=g, dtype=torch.float64))
        keys = torch.unique(torch.cat([keys, doc * D + term_of[r.clamp_(max=D - 1)]]))
        need = want - torch.bincount(torch.div(keys, D, rounding_mode="floor"), minlength=N)
    doc = torch.div(keys, D, rounding_mode="floor")
    term = keys - doc * D
    del keys
    df = torch.bincount(term, minlength=D).to(torch.float64)
    tf = 1.0 + torch.poisson(torch.ones(term.numel(), device=dev), generator=g).to(torch.float64)
    v = tf * torch.log(N / df[term])
    keep = v > 0
    if not bool(keep.all()):
        doc, term, v = doc[keep], term[keep], v[keep]
    # squared norms in whole numbers, so that they do not depend on the order of the sum
    ss = torch.zeros(N, dtype=torch.int64, device=dev).index_add_(0, doc, (v * v * 2.0**24).round().to(torch.int64))
    val = (v / torch.sqrt(ss[doc].to(torch.float64) * 2.0**-24)).to(torch.float32)
    row_ptr = torch.zeros(N + 1, dtype=torch.int64, device=dev)
    row_ptr[1:] = torch.bincount(doc, minlength=N).cumsum(0)
    return row_ptr, term.to(torch.int32), val


def _case_corpus(c, seed):
    return _corpus(c["N"], c["D"], c["s"], c["mean"], c["sigma"], seed)


def _seeds(N, k, seed):
    g = torch.Generator().manual_seed(seed + 7919)
    return np.ascontiguousarray(torch.randperm(N, generator=g)[:k].to(torch.int32).numpy())


def _batch_instances(c):
    """Sizes (N, D, k, mean length) of the instances: N, D and k log-uniform, mean length uniform."""
    rng = random.Random(c["sizes"])
    out = []
    for _ in range(c["n_inst"]):
        N = max(64, int(_log_uniform(rng, 5_000, 200_000) * c["scale"]))
        D = int(_log_uniform(rng, 20_000, 100_000))
        k = max(2, min(int(_log_uniform(rng, 16, 2_000) * math.sqrt(c["scale"])), N // 8))
        out.append((N, D, k, rng.uniform(30.0, 250.0)))
    return out


def _labelings(c, seed):
    """Two labelings with every cluster in use, different in a part of the objects."""
    N, k = c["N"], c["k"]
    g = torch.Generator().manual_seed(seed + 104729)
    a = (torch.randperm(N, generator=g) % k).to(torch.int32)
    change = torch.rand(N, generator=g) < c["change"]
    change[:k] = False
    a[:k] = torch.arange(k, dtype=torch.int32)
    b = torch.where(change, torch.randint(0, k, (N,), generator=g, dtype=torch.int32), a)
    return a, b


def _centroid_entries(c, seed):
    """Cluster-major centroids of random sparse rows, and which clusters are invariant (numpy)."""
    rng = np.random.default_rng(seed)
    k, D, n = c["k"], c["D"], c["entries"]
    # Zipf-like terms, distinct inside a row
    p = np.arange(1, D + 1, dtype=np.float64) ** -0.8
    cdf = np.cumsum(p) / p.sum()
    keys = np.empty(0, dtype=np.int64)
    for rounds in range(1000):  # repeats are drawn again, from all terms alike when many rounds left some
        m = n - len(keys)
        if m <= 0:
            break
        t = np.minimum(np.searchsorted(cdf, rng.random(m)), D - 1) if rounds < 10 else rng.integers(0, D, m)
        keys = np.unique(np.concatenate([keys, rng.integers(0, k, m) * np.int64(D) + t]))
    clu, term = keys // D, (keys % D).astype(np.int32)
    off = np.zeros(k + 1, dtype=np.int64)
    off[1:] = np.cumsum(np.bincount(clu, minlength=k))
    u = (rng.random(len(keys)) * 0.2 + 1e-4).astype(np.float32)
    lam = (rng.random(k) < 0.5).astype(np.uint8)
    return off, term, u, lam


def _capacity(N, mean):
    """Room for the centroids: at most one entry per object non-zero, and some for clusters that emptied."""
    return int(N * mean + 8 * mean * math.sqrt(N)) + 4_096


class _Centroids:
    """Pinned host buffers for the centroids, kept from call to call (zero beyond the entries)."""

    def __init__(self, k, cap):
        self.off = torch.zeros(k + 1, dtype=torch.int64, pin_memory=True)
        self.term = torch.zeros(cap, dtype=torch.int32, pin_memory=True)
        self.u = torch.zeros(cap, dtype=torch.float32, pin_memory=True)

    def get(self, ctx):
        import ctypes
        n = ctypes.c_int64(0)
        st = S.load().sivf_get_centroids(ctx, self.off.data_ptr(), self.term.data_ptr(), self.u.data_ptr(),
                                         self.term.numel(), ctypes.byref(n))
        if st != S.SIVF_OK:
            raise RuntimeError(f"sivf_get_centroids: {S.STATUS_NAMES[st]}")
        return {"nnz": n.value, "off": self.off, "term": self.term, "u": self.u}


def prepare(case, seed):
    c, kind = case, case["kind"]
    st = SimpleNamespace(case=c, kind=kind)
    if kind == "build":
        off, term, u, lam = _centroid_entries(c, seed)
        dev = torch.device("cuda")
        st.n = len(term)
        st.inputs = [torch.from_numpy(a).to(dev) for a in (off, term, u, lam)]
        st.out = [torch.empty(c["D"] + 1, dtype=torch.int64, device=dev),
                  torch.empty(c["D"], dtype=torch.int32, device=dev),
                  torch.empty(st.n, dtype=torch.int32, device=dev),
                  torch.empty(st.n, dtype=torch.float32, device=dev)]
        S.load()
        return st
    if kind == "batch":
        inst = _batch_instances(c)
        corpora, ini = [], []
        for m, (N, D, k, mean) in enumerate(inst):
            sd = seed * 1000 + m
            rp, ix, vl = _corpus(N, D, 1.1, mean, 0.7, sd)
            corpora.append(SimpleNamespace(row_ptr=rp.cpu().numpy(), idx=ix.cpu().numpy(), val=vl.cpu().numpy(), D=D))
            ini.append(_seeds(N, k, sd))
        ks = [i[2] for i in inst]
        st.g = SIVFBatch(corpora, ks, ini, precision=c["precision"], icp=c["icp"], use_graph=c["graph"])
        base = np.cumsum([0] + [i[0] for i in inst[:-1]])
        st.ini = np.ascontiguousarray(np.concatenate([a + b for a, b in zip(ini, base)]), dtype=np.int32)
        st.cen = _Centroids(sum(ks), sum(_capacity(i[0], i[3]) for i in inst))
        return st
    rp, ix, vl = _case_corpus(c, seed)
    st.ini = _seeds(c["N"], c["k"], seed)
    st.cen = _Centroids(c["k"], _capacity(c["N"], c["mean"]))
    st.labels = torch.empty(c["N"], dtype=torch.int32, device="cuda")
    st.g = SIVF(rp, ix, vl, c["D"], c["k"], st.ini, precision=c["precision"], icp=c.get("icp", 1),
                use_graph=c.get("graph", False))
    if kind == "resume":  # the saved labels
        st.g.run(c["done"])
        st.saved = st.g.labels_device()
    elif kind == "update":
        st.a, st.b = (x.cuda() for x in _labelings(c, seed))
    return st


# ---------------------------------------------------------------- one pass

def run(st):
    c, kind = st.case, st.kind
    if kind == "build":
        off, term, u, lam = st.inputs
        S.sivf_build_inverted_file_noalloc(c["k"], c["D"], st.n, off.data_ptr(), term.data_ptr(), u.data_ptr(),
                                           lam.data_ptr(), *[o.data_ptr() for o in st.out],
                                           torch.cuda.current_stream().cuda_stream)
        return {"off": st.out[0], "mf0": st.out[1], "cid": st.out[2], "u": st.out[3]}
    if kind == "batch":
        S.sivf_reseed(st.g.ctx, st.ini.ctypes.data)
        iters, objective = st.g.run(c["iters"])
        labels = [st.g.labels(m) for m in range(st.g.n_inst)]
        return {"labels": np.concatenate(labels), "iters": iters, "objective": objective, **st.cen.get(st.g.ctx)}
    if kind == "update":
        st.g.set_labels(st.a)
        st.g.update()
        st.g.set_labels(st.b)
        st.g.update()
        return st.cen.get(st.g.ctx)
    st.g.reseed(st.ini)
    if kind == "resume":
        st.g.set_labels(st.saved)
        st.g.update()
    iters, objective = st.g.run(c["iters"])
    return {"labels": st.g.labels_device(st.labels), "iters": iters, "objective": objective, **st.cen.get(st.g.ctx)}


# ---------------------------------------------------------------- the work

def _zipf_model(N, D, k, s, mean):
    """(postings of an object's lists with seed centroids, and with means; centroid
    non-zeros of the means), expected for Zipf documents of this mean length."""
    r = np.arange(1, D + 1, dtype=np.float64) ** -s
    lo, hi = 0.0, 1e12
    for _ in range(100):  # P(term in document) = 1 - exp(-c r^-s), with c giving the mean length
        mid = (lo + hi) / 2 if hi < 1e11 else lo * 2 + 1
        if (1.0 - np.exp(-mid * r)).sum() > min(mean, D * 0.9):
            hi = mid
        else:
            lo = mid
        if hi < 1e11 and hi - lo < 1e-6 * hi:
            break
    p = 1.0 - np.exp(-hi * r)
    q = 1.0 - (1.0 - np.minimum(p, 1 - 1e-12)) ** (N / k)
    return k * float((p * p).sum()), k * float((p * q).sum()), k * float(q.sum())


def _run_work(N, D, k, s, mean, first, means):
    """Bytes and flops of `first` iterations over seed centroids and `means` over means:
    per iteration the corpus read, labels and centroids written, one multiply-add per posting."""
    p0, p1, cn = _zipf_model(N, D, k, s, mean)
    nnz = N * mean
    it = first + means
    return it * (8.0 * nnz + 12.0 * N + 8.0 * cn), 2.0 * N * (first * p0 + means * p1)


def work(case):
    c, kind = case, case["kind"]
    if kind == "build":  # entries in and out, offsets and front lengths
        return {"bytes": 16.0 * c["entries"] + 9.0 * c["k"] + 12.0 * c["D"], "flops": 0}
    if kind == "batch":
        b = f = 0.0
        for N, D, k, mean in _batch_instances(c):
            x, y = _run_work(N, D, k, 1.1, mean, 1, min(3, c["iters"] - 1))
            b, f = b + x, f + y
        return {"bytes": b, "flops": f}
    if kind == "update":  # the changed objects and the labels in, the centroids out, twice
        _, _, cn = _zipf_model(c["N"], c["D"], c["k"], c["s"], c["mean"])
        nnz = c["N"] * c["mean"] * c["change"]
        return {"bytes": 2.0 * (8.0 * nnz + 4.0 * c["N"] + 8.0 * cn), "flops": 4.0 * nnz}
    if kind == "resume":  # one scan of every list; what the filter leaves after that is small
        b, f = _run_work(c["N"], c["D"], c["k"], c["s"], c["mean"], 0, 1)
        return {"bytes": b * c["iters"], "flops": f}
    b, f = _run_work(c["N"], c["D"], c["k"], c["s"], c["mean"], 1, c["iters"] - 1)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------- 64-bit values

def _exact_means(N, D, k, rp, ix, vl, labels, old):
    """Dense float64 unit means of the clusters; empty clusters keep theirs."""
    doc = torch.repeat_interleave(torch.arange(N, device=rp.device), rp[1:] - rp[:-1])
    m = torch.zeros(k * D, dtype=torch.float64, device=rp.device)
    m.index_add_(0, labels.long()[doc] * D + ix.long(), vl.double())
    m = m.view(k, D)
    norm = m.norm(dim=1, keepdim=True)
    out = torch.where(norm > 0, m / norm.clamp(min=1e-300), old)
    return out, float(norm.sum())


def _values(m, cap):
    """The non-zero values of the rows, in the room that the case has for them."""
    u = torch.zeros(cap, dtype=torch.float64, device=m.device)
    nz = m[m != 0]
    u[:nz.numel()] = nz
    return u


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "build":
        off, term, u, lam = _centroid_entries(c, seed)
        clu = np.repeat(np.arange(c["k"]), np.diff(off))
        order = np.lexsort((clu, lam[clu], term))
        lens = np.bincount(term, minlength=c["D"])
        return {"off": np.concatenate([[0], np.cumsum(lens)]),
                "mf0": np.bincount(term[lam[clu] == 0], minlength=c["D"]).astype(np.int32),
                "cid": clu[order].astype(np.int32), "u": u[order].astype(np.float64)}
    if kind == "batch" or kind == "resume":  # many iterations of several corpora, or from labels of the library
        return None
    N, D, k = c["N"], c["D"], c["k"]
    if kind == "update":
        if float(k) * D > 5e8:
            return None
        rp, ix, vl = _case_corpus(c, seed)
        b = _labelings(c, seed)[1].cuda()
        m, _ = _exact_means(N, D, k, rp, ix, vl, b, torch.zeros(k, D, dtype=torch.float64, device="cuda"))
        return {"nnz": None, "off": None, "term": None, "u": _values(m, _capacity(N, c["mean"]))}
    if float(N) * D > 3e7 or float(N) * k * c["iters"] > 1e8:
        return None
    rp, ix, vl = _case_corpus(c, seed)
    doc = torch.repeat_interleave(torch.arange(N, device=rp.device), rp[1:] - rp[:-1])
    x = torch.zeros(N, D, dtype=torch.float64, device=rp.device)
    x[doc, ix.long()] = vl.double()
    m = x[torch.from_numpy(_seeds(N, k, seed)).long().cuda()].clone()
    prev, objective, done = None, 0.0, 0
    for done in range(1, c["iters"] + 1):
        a = torch.from_numpy(np.argmax((x @ m.T).cpu().numpy(), axis=1)).cuda()
        if prev is not None and bool((a == prev).all()):
            break
        m, objective = _exact_means(N, D, k, rp, ix, vl, a, m)
        prev = a
    return {"labels": None, "iters": None, "objective": objective, "nnz": None, "off": None, "term": None,
            "u": _values(m, _capacity(N, c["mean"]))}
