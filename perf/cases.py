"""Measured cases: the benchmark programs of the framework, issued through its
public classes (``gdag.Context`` and ``workloads``) as a user's program issues
them, over the range of sizes that the serving workload draws from (1/64 of the
full size up to the full size).

A state is one long-running program: a context that retires completed work
without host waits, its arrays resident in device memory, and the program's
recorded step.  One pass is one step of the program."""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2012_09646_gb300 import gdag as G
from paper_2012_09646_gb300 import workloads as W

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # VEC at 1/64 of its full length: a short request whose host writes
        # two vectors and reads one sum back; latency and launches
        {"name": "vec-small", "kind": "vec", "n": 15_625},
        # VEC at its full length
        {"name": "vec-full", "kind": "vec", "n": 1_000_000},
        # ten small option books, a length that no vector width divides
        {"name": "bs-small", "kind": "bs", "n": 156_253, "count": 10},
        # ten full option books: the headline workload
        {"name": "bs-full", "kind": "bs", "n": 10_000_000, "count": 10},
        # the image program at 1/64 of its full area
        {"name": "img-small", "kind": "img", "rows": 512, "cols": 512},
        # an image whose rows are not a multiple of four pixels
        {"name": "img-ragged", "kind": "img", "rows": 1300, "cols": 3001},
        # the full image
        {"name": "img-full", "kind": "img", "rows": 4096, "cols": 4096},
        # the classifier ensemble on a short batch of narrow rows: a feature
        # count that is not a multiple of 64, an odd number of rows
        {"name": "ml-narrow", "kind": "ml", "rows": 4097, "feats": 96, "classes": 12},
        # the classifier ensemble on its full batch
        {"name": "ml-full", "kind": "ml", "rows": 100_000, "feats": 1024, "classes": 10},
        # hubs and authorities of a batch of small graphs in one program
        {"name": "hits-batch", "kind": "hits_batch", "count": 64, "nmin": 10_000, "nmax": 100_000},
        # hubs and authorities of the full graph
        {"name": "hits-full", "kind": "hits", "n": 10_000_000, "nnz": 50_000_000},
        # the two-branch convolution network on its full batch
        {"name": "dl-full", "kind": "dl", "n": 16, "h": 256, "w": 256},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["vec", "bs", "img", "img", "ml", "ml", "hits", "hits_batch", "dl"])
    if kind == "vec":
        return {"kind": kind, "n": _log_int(rng, 15_625, 1_000_000)}
    if kind == "bs":
        return {"kind": kind, "n": _log_int(rng, 156_250, 10_000_000), "count": rng.randint(6, 10)}
    if kind == "img":
        return {"kind": kind, "rows": _log_int(rng, 500, 4096), "cols": _log_int(rng, 500, 4096)}
    if kind == "ml":
        return {"kind": kind, "rows": _log_int(rng, 1_563, 100_000),
                "feats": rng.choice([96, 192, 256, 352, 512, 640, 1024]), "classes": rng.randint(2, 16)}
    if kind == "hits":
        n = _log_int(rng, 156_250, 8_000_000)
        return {"kind": kind, "n": n, "nnz": 5 * n}
    if kind == "hits_batch":
        nmin = _log_int(rng, 5_000, 20_000)
        return {"kind": kind, "count": rng.randint(8, 64), "nmin": nmin, "nmax": rng.randint(2, 8) * nmin}
    return {"kind": kind, "n": rng.randint(1, 16), "h": 2 * rng.randint(32, 128), "w": 8 * rng.randint(8, 32)}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _rand(shape, g, lo=0.0, hi=1.0):
    return torch.rand(shape, generator=g, device=DEV, dtype=torch.float32) * (hi - lo) + lo


def _dyadic(t):
    """Multiples of 1/256 below 1000/256: tables whose scores are exact."""
    return ((t.double() * 256.0).round().clamp(-999, 999) / 256.0).float()


def _vec(case, seed):
    g = _gen(seed)
    return _rand(case["n"], g), _rand(case["n"], g)


def _bs(case, seed):
    g = _gen(seed)
    return [_rand(case["n"], g, 10.0, 100.0) for _ in range(case["count"])]


def _img(case, seed):
    return _rand((case["rows"], case["cols"]), _gen(seed))


def _ml(case, seed):
    g = _gen(seed)
    f, k = case["feats"], case["classes"]
    X = torch.randint(0, 16, (case["rows"], f), generator=g, device=DEV, dtype=torch.int32)
    # class-conditional feature probabilities (Dirichlet(2): sums of two
    # exponentials, normalised over the features) and their centred logs
    e = -torch.log1p(-torch.rand((2, f, k), generator=g, device=DEV, dtype=F64)).sum(0) + 1e-9
    logp = torch.log(e / e.sum(0, keepdim=True))
    nb = _dyadic(logp - logp.mean(1, keepdim=True))
    prior = torch.log(torch.rand(k, generator=g, device=DEV, dtype=F64) + 0.1)
    w = _dyadic(torch.randn((f, k), generator=g, device=DEV) * 0.05)
    b = _dyadic(torch.randn(k, generator=g, device=DEV) * 0.5)
    return X, nb, _dyadic(prior - prior.mean()), w, b


def _graph(n, nnz, g):
    """CSR of A and of its transpose as (rowptr, col, val) on the device:
    power-law out-degrees (exponent 2.1) with exactly nnz edges, uniform
    destinations, no self-loops, no duplicate edges, unit weights."""
    u = 1.0 - torch.rand(n, generator=g, device=DEV, dtype=F64)
    d = torch.floor(u ** (-1.0 / 1.1)).clamp_(max=n - 1)
    d = torch.floor(d * (nnz / d.sum())).clamp_(max=n - 1).long()
    while (short := nnz - int(d.sum())) > 0:
        room = torch.nonzero(d < n - 1).flatten()
        pick = room[torch.randperm(room.numel(), generator=g, device=DEV)[:short]]
        d[pick] += 1
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), d, output_size=nnz)
    cols = torch.randint(0, n - 1, (nnz,), generator=g, device=DEV)
    cols += cols >= rows
    key = (rows * n + cols).sort().values
    while True:  # duplicates get new destinations
        dup = torch.nonzero(key[1:] == key[:-1]).flatten() + 1
        if dup.numel() == 0:
            break
        r = key[dup] // n
        c = torch.randint(0, n - 1, (dup.numel(),), generator=g, device=DEV)
        key[dup] = r * n + c + (c >= r)
        key = key.sort().values
    rows, cols = key // n, key % n
    tkey = (cols * n + rows).sort().values

    def csr(k):
        ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
        ptr[1:] = torch.cumsum(torch.bincount(k // n, minlength=n), 0)
        return ptr.int(), (k % n).int(), torch.ones(nnz, dtype=torch.float32, device=DEV)

    return csr(key), csr(tkey)


def _graphs(case, seed):
    g = _gen(seed)
    if case["kind"] == "hits":
        return [_graph(case["n"], case["nnz"], g)]
    return [_graph(n, 5 * n, g) for n in _batch_sizes(case)]


def _batch_sizes(case):
    """Vertex counts log-uniform on [nmin, nmax], the same for every seed."""
    r = np.random.default_rng(case["nmin"])
    return [int(v) for v in np.exp(r.uniform(math.log(case["nmin"]), math.log(case["nmax"]), case["count"]))]


def _dl(case, seed):
    g = _gen(seed)
    n, h, w = case["n"], case["h"], case["w"]
    q = lambda t: t.bfloat16().float()  # noqa: E731
    nrm = lambda shape, s: torch.randn(shape, generator=g, device=DEV) * s  # noqa: E731
    x1, x2 = q(_rand((n, 3, h, w), g)), q(_rand((n, 3, h, w), g))
    w1, w2 = q(nrm((64, 3, 3, 3), 0.3)), q(nrm((64, 3, 3, 3), 0.3))
    return x1, x2, w1, nrm(64, 0.1), w2, nrm(64, 0.1), nrm((128, 10), 0.1), nrm(10, 0.1)


# ------------------------------------------------------------------- passes
def prepare(case, seed):
    ctx = G.Context(retire_by_query=True)
    kind = case["kind"]
    if kind == "vec":
        d = W.VecDag(ctx, case["n"])
        d.load(*(t.cpu() for t in _vec(case, seed)))
    elif kind == "bs":
        d = W.BsDag(ctx, case["n"], count=case["count"], host=False)
        d.load_device(_bs(case, seed))
    elif kind == "img":
        d = W.ImgDag(ctx, case["rows"], case["cols"])
        d.img.copy_(_img(case, seed).reshape(-1))
    elif kind == "ml":
        d = W.MlDag(ctx, case["rows"], case["feats"], case["classes"])
        d.load(*_ml(case, seed))
    elif kind == "hits":
        d = W.HitsDag(ctx, *_graphs(case, seed)[0])
        d.run(iters=0, read=False)  # a = h = 1
    elif kind == "hits_batch":
        cpu = lambda m: tuple(t.cpu().numpy() for t in m)  # noqa: E731
        d = W.HitsBatchDag(ctx, [(cpu(a), cpu(t)) for a, t in _graphs(case, seed)])
        d.run(iters=0, read=False)
    else:
        d = W.DlDag(ctx, case["n"], case["h"], case["w"])
        d.load(*_dl(case, seed))
    ctx.sync()
    torch.cuda.synchronize()
    return {"kind": kind, "dag": d}


def run(state):
    kind, d = state["kind"], state["dag"]
    if kind == "vec":  # the host writes both vectors and reads the sum
        z = d.step()
        return {"z": z, "x": d.x, "y": d.y}
    if kind == "bs":
        d.step_resident()
        return {"c%d" % i: c for i, c in enumerate(d.C)}
    if kind == "img":
        d.launch_all()
        return {"out": d.out, "s": d.s, "b5": d.b5, "b9": d.b9, "e5": d.e5, "e9": d.e9, "mm5": d.mm5, "mm9": d.mm9}
    if kind == "ml":
        d.launch_all()
        return {"p1": d.S1, "p2": d.S2, "labels": d.labels}
    if kind == "dl":
        d.launch_all()
        return {"logits": d.logits, "e1": d.e1, "e2": d.e2, "p1": d.p1, "p2": d.p2, "status": d.status}
    # HITS: five iterations over alternating buffers
    cur, nxt = ("a", "h"), ("a2", "h2")
    for _ in range(5):
        d.iterate(cur[0], cur[1], nxt[0], nxt[1])
        cur, nxt = nxt, cur
    return {"a": d.vec["a2"], "h": d.vec["h2"]}


def work(case):
    """Each input read once and each output written once; HITS reads its
    matrices and vectors once per iteration."""
    kind = case["kind"]
    if kind == "vec":
        return {"bytes": 16 * case["n"] + 4, "flops": 4 * case["n"]}
    if kind == "bs":
        return {"bytes": 8 * case["n"] * case["count"], "flops": 40 * case["n"] * case["count"]}
    if kind == "img":
        n = case["rows"] * case["cols"]
        return {"bytes": 4 * n * 7, "flops": 100 * n}
    if kind == "ml":
        r, f, k = case["rows"], case["feats"], case["classes"]
        return {"bytes": 4 * r * f + 8 * r * k + 4 * r + 8 * f * k, "flops": 4 * r * f * k}
    if kind == "dl":
        px = case["n"] * case["h"] * case["w"]
        return {"bytes": 2 * (2 * 3 * px + 2 * 64 * px // 4), "flops": 2 * 2 * 27 * 64 * px}
    if kind == "hits":
        n, nnz = case["n"], case["nnz"]
    else:
        n = sum(_batch_sizes(case))
        nnz = 5 * n
    return {"bytes": 5 * 2 * (8 * nnz + 12 * n), "flops": 5 * 2 * (2 * nnz + 3 * n)}


# ------------------------------------------------- the same in 64 bits
def exact(case, seed):
    kind = case["kind"]
    if kind == "vec":
        x, y = (t.double() ** 2 for t in _vec(case, seed))
        return {"z": float((x - y).sum()), "x": x, "y": y}
    if kind == "bs":
        K, r, sg, T = 60.0, 0.1, 0.2, 1.0
        f32 = lambda v: float(np.float32(v))  # noqa: E731 (the parameters are float32)
        K, r, sg, T = f32(K), f32(r), f32(sg), f32(T)
        out = {}
        for i, s in enumerate(_bs(case, seed)):
            s = s.double()
            d1 = (torch.log(s / K) + (r + sg * sg / 2) * T) / (sg * math.sqrt(T))
            cdf = lambda v: 0.5 * torch.erfc(-v / math.sqrt(2.0))  # noqa: E731
            out["c%d" % i] = s * cdf(d1) - K * math.exp(-r * T) * cdf(d1 - sg * math.sqrt(T))
        return out
    if kind == "img":
        return _img_exact(_img(case, seed).double())
    if kind == "ml":
        X, t1, b1, t2, b2 = _ml(case, seed)
        p = []
        for t, b in ((t1, b1), (t2, b2)):
            s = torch.cat([x.double() @ t.double() for x in X.split(16384)]) + b.double()
            p.append(torch.softmax(s, 1))
        return {"p1": p[0], "p2": p[1], "labels": None}
    if kind == "dl":
        return _dl_exact(*_dl(case, seed))
    outs = [_hits_exact(*m) for m in _graphs(case, seed)]
    return {"a": torch.cat([o[0] for o in outs]), "h": torch.cat([o[1] for o in outs])}


def _taps(radius, sigma):
    w = [math.exp(-(k * k) / (2.0 * sigma * sigma)) for k in range(-radius, radius + 1)]
    return [float(np.float32(v / sum(w))) for v in w]  # the filter's taps are float32


def _shift(t, dy, dx):
    """t with rows moved by dy and columns by dx, edge pixels repeated."""
    r = (torch.arange(t.shape[0], device=t.device) + dy).clamp_(0, t.shape[0] - 1)
    c = (torch.arange(t.shape[1], device=t.device) + dx).clamp_(0, t.shape[1] - 1)
    t = t[r] if dy else t
    return t[:, c] if dx else t


def _img_exact(im):
    def blur(radius, sigma):
        w = _taps(radius, sigma)
        v = sum(wk * _shift(im, k - radius, 0) for k, wk in enumerate(w))
        return sum(wk * _shift(v, 0, k - radius) for k, wk in enumerate(w))

    def sobel(t):
        sv = _shift(t, -1, 0) + 2 * t + _shift(t, 1, 0)
        dv = _shift(t, 1, 0) - _shift(t, -1, 0)
        gx = _shift(sv, 0, 1) - _shift(sv, 0, -1)
        gy = _shift(dv, 0, -1) + 2 * dv + _shift(dv, 0, 1)
        return torch.sqrt(gx * gx + gy * gy)

    b5, b9 = blur(2, 1.0), blur(4, 2.0)
    r5, r9 = sobel(b5), sobel(b9)
    mm = [torch.stack([e.min(), e.max()]) for e in (r5, r9)]
    e5, e9 = ((e - m[0]) / (m[1] - m[0]) for e, m in zip((r5, r9), mm))
    s = im + 0.5 * (im - b5)
    out = e5 * s + (1 - e5) * (e9 * b5 + (1 - e9) * b9)
    f = lambda t: t.reshape(-1)  # noqa: E731
    return {"out": f(out), "s": f(s), "b5": f(b5), "b9": f(b9), "e5": f(e5), "e9": f(e9), "mm5": mm[0], "mm9": mm[1]}


def _hits_exact(A, AT):
    n = A[0].numel() - 1

    def rows_of(m):
        return torch.repeat_interleave(torch.arange(n, device=DEV), m[0].long().diff(), output_size=m[1].numel())

    def spmv(m, rows, x):
        return torch.zeros(n, dtype=F64, device=DEV).index_add_(0, rows, m[2].double() * x[m[1].long()])

    ra, rt = rows_of(A), rows_of(AT)
    a = torch.ones(n, dtype=F64, device=DEV)
    h = torch.ones(n, dtype=F64, device=DEV)
    for _ in range(5):
        a, h = spmv(AT, rt, h), spmv(A, ra, a)
        a, h = a / a.norm().clamp_min(1e-300), h / h.norm().clamp_min(1e-300)
    return a, h


def _dl_exact(x1, x2, w1, b1, w2, b2, wd, bd):
    def branch(x, w, b):
        # the convolution as 27 shifted products, image by image
        n, _, hh, ww = x.shape
        out = []
        for im in x.double():
            p = torch.nn.functional.pad(im, (1, 1, 1, 1))
            taps = torch.stack([p[c, i:i + hh, j:j + ww] for c in range(3) for i in range(3) for j in range(3)])
            y = (w.double().reshape(64, 27) @ taps.reshape(27, -1)).reshape(64, hh, ww) + b.double().reshape(64, 1, 1)
            out.append(torch.nn.functional.max_pool2d(y.clamp_min(0)[None], 2)[0])
        return torch.stack(out)

    p1, p2 = branch(x1, w1, b1), branch(x2, w2, b2)
    e1, e2 = p1.mean((2, 3)), p2.mean((2, 3))
    logits = torch.cat([e1, e2], 1) @ wd.double() + bd.double()
    return {"logits": logits, "e1": e1, "e2": e2, "p1": p1, "p2": p2, "status": None}
