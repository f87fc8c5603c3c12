"""Workloads that stand for the use of this library, for timing it and comparing its results.

Each case is one call of a public entry point on device-resident inputs, as a user's program
makes it: the cost matrix stays in `w`, each pass restores it into the work matrix and closes
that in place (the closures overwrite their input).  Graphs are directed Erdos-Renyi graphs, as
everywhere in this repository (integer weights uniform in [1, wmax], or float32 lognormal(0, 1));
missing edges hold the sentinel (0x3FFFFFFF, or +inf).  Matrices are plain contiguous tensors, so an
odd n gives rows that are not 16-byte aligned.
"""
import math

import numpy as np
import torch

import paper_2310_03983_gb300 as apsp

INF = apsp.APSP_INF_I32
DTYPES = {"i32": torch.int32, "f32": torch.float32}


def listed():
    return [
        # The smallest graphs of a request stream: one tile, so the call is launches and latency.
        dict(name="fw_i32_n100", kind="fw", dtype="i32", n=100, p=0.2, wmax=100),
        # The small single-graph configuration: a few dependent block steps, far too little work for
        # every SM.
        dict(name="fw_i32_n512", kind="fw", dtype="i32", n=512, p=0.1, wmax=100),
        # A mid-size request with real-valued costs and an odd, unaligned size.
        dict(name="fw_f32_n1237", kind="fw", dtype="f32", n=1237, p=0.1, wmax=0),
        # The mid-size configuration: dense, integer costs.
        dict(name="fw_i32_n4096", kind="fw", dtype="i32", n=4096, p=0.5, wmax=1000),
        # The largest request of the serving configuration, real-valued costs.
        dict(name="fw_f32_n8192", kind="fw", dtype="f32", n=8192, p=0.05, wmax=0),
        # The headline benchmark: one large sparse graph with small integer costs.
        dict(name="fw_i32_n32768", kind="fw", dtype="i32", n=32768, p=0.05, wmax=100),
        # The recursive closure on the mid-size configuration, with its default cutoff.
        dict(name="rkleene_i32_n4096", kind="rkleene", dtype="i32", n=4096, p=0.5, wmax=1000, cutoff=0),
        # The batch configuration: 2048 graphs of uneven size in one call.
        dict(name="batch_i32_2048", kind="batch", dtype="i32", count=2048, n_lo=32, n_hi=1024, wmax=100),
        # What the server admits at once: a few small real-valued graphs closed in one call.
        dict(name="batch_f32_16", kind="batch", dtype="f32", count=16, n_lo=64, n_hi=1024, wmax=0),
        # A (min,+) product of two distance tables, ragged and unaligned.
        dict(name="gemm_f32_ragged", kind="gemm", dtype="f32", m=3001, n=2503, k=1999, wmax=0),
        # Path recovery after a closure, real-valued costs.
        dict(name="pred_f32_n3000", kind="pred", dtype="f32", n=3000, p=0.1, wmax=0),
        # The paper's own method, repeated squaring, at its largest graph size.
        dict(name="squaring_i32_n1024", kind="squaring", dtype="i32", n=1024, p=0.4, wmax=100),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["fw", "batch", "rkleene", "gemm", "pred", "squaring", "signed", "cta"],
                       [8, 3, 2, 2, 2, 1, 1, 1])[0]
    c = dict(kind=kind, dtype=rng.choice(["i32", "f32"]))
    c["wmax"] = rng.choice([100, 100, 1000, 1000000]) if c["dtype"] == "i32" else 0
    p = round(math.exp(rng.uniform(math.log(0.01), math.log(0.5))), 4)
    if kind == "gemm":
        c.update(m=_log(rng, 100, 6000), n=_log(rng, 100, 6000), k=_log(rng, 100, 6000))
    elif kind == "batch":
        c.update(count=_log(rng, 8, 1500), n_lo=rng.randint(16, 128), n_hi=rng.randint(300, 1200))
        c["wmax"] = min(c["wmax"], 1000)
    else:
        top = dict(fw=12288, rkleene=8192, pred=5000, squaring=3000, signed=4000, cta=1024)[kind]
        n = _log(rng, 64, top)
        if rng.random() < 0.5:  # half of them on whole 16-byte rows
            n = max(4, n // 4 * 4)
        c.update(n=n, p=p)
        if kind == "rkleene":
            c["cutoff"] = rng.choice([0, 1024])
        if kind == "signed":
            c["wmax"] = min(c["wmax"], 1000)
    return c


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(0x41505350 + int(seed))


def _weights(shape, c, p, g):
    """Random costs: each entry is an edge with probability p (a number, or one per entry)."""
    if c["dtype"] == "i32":
        w = torch.randint(1, c["wmax"] + 1, shape, generator=g, device="cuda", dtype=torch.int32)
        none = INF
    else:
        w = torch.empty(shape, device="cuda").log_normal_(0.0, 1.0, generator=g)
        none = math.inf
    # in slices: the variates of the largest matrix would take as much again as the matrix
    flat, prob = w.view(-1), p if isinstance(p, torch.Tensor) else None
    step = 1 << 28
    for a in range(0, flat.numel(), step):
        s = flat[a:a + step]
        u = torch.rand(s.shape, generator=g, device="cuda")
        s.masked_fill_(u >= (p if prob is None else prob[a:a + step]), none)
    return w


def _graph(c, seed):
    w = _weights((c["n"], c["n"]), c, c["p"], _gen(seed))
    w.fill_diagonal_(0)
    return w


def _batch_layout(c):
    """Sizes and densities of a batch (n log-uniform, p uniform in [0.02, 0.8]; the same for every
    seed) and the pool layout apsp_batched documents: rows padded to 16 bytes, graphs one after
    the other."""
    rng = np.random.default_rng([c["count"], c["n_lo"], c["n_hi"], 0x42415443])
    ns = np.rint(np.exp(rng.uniform(math.log(c["n_lo"]), math.log(c["n_hi"]), c["count"]))).astype(np.int32)
    ps = rng.uniform(0.02, 0.8, c["count"]).astype(np.float32)
    lds = (ns + 3) // 4 * 4
    sizes = ns.astype(np.int64) * lds
    offsets = np.concatenate([[0], np.cumsum(sizes)[:-1]]).astype(np.int64)
    return ns, ps, lds.astype(np.int32), offsets, sizes


def _batch_pool(c, seed):
    ns, ps, lds, offsets, sizes = _batch_layout(c)
    dev = [torch.from_numpy(x).cuda() for x in (ns, ps, lds, offsets, sizes)]
    total = int(sizes.sum())
    p = torch.repeat_interleave(dev[1], dev[4], output_size=total)
    pool = _weights((total,), c, p, _gen(seed))
    return pool, ns, dev


def _torch_closure(w, dtype):
    """Eq. 1 vertex by vertex in the given type (missing edges +inf, or the sentinel)."""
    d = w.clone() if w.dtype == dtype else w.to(dtype)
    t = torch.empty_like(d)
    for k in range(d.shape[-1]):
        torch.add(d[..., :, k:k + 1], d[..., k:k + 1, :], out=t)
        torch.minimum(d, t, out=d)
    return d


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "gemm":
        g = _gen(seed)
        a, b = (_weights(s, c, 0.9, g) for s in ((c["m"], c["k"]), (c["k"], c["n"])))
        return dict(case=c, a=a, b=b, out=torch.empty((c["m"], c["n"]), dtype=a.dtype, device="cuda"))
    if kind == "batch":
        pool, ns, (d_ns, _, d_lds, d_offsets, _) = _batch_pool(c, seed)
        order = torch.from_numpy(np.argsort(-ns, kind="stable").astype(np.int32)).cuda()
        ws = torch.empty(apsp.apsp_batched_staged_workspace_bytes(ns, pool.dtype), dtype=torch.uint8, device="cuda")
        return dict(case=c, w=pool, d=torch.empty_like(pool), ns_host=ns, ns=d_ns, lds=d_lds, offsets=d_offsets,
                    order=order, ws=ws)
    w = _graph(c, seed)
    if kind == "signed":  # costs shifted by a potential: negative edges, but no negative cycle
        g = _gen(seed + 1000003)
        n = c["n"]
        if c["dtype"] == "i32":
            pot = torch.randint(0, 81, (n,), generator=g, device="cuda", dtype=torch.int32)
            w = torch.where(w < INF, w + pot[:, None] - pot[None, :], w)
        else:
            pot = torch.rand(n, generator=g, device="cuda") * 30.0
            w = w + pot[:, None] - pot[None, :]
        w.fill_diagonal_(0)
    if kind == "pred":
        d = _torch_closure(w, w.dtype)
        return dict(case=c, w=w, d=d.clamp_(max=INF) if c["dtype"] == "i32" else d,
                    pred=torch.empty((c["n"], c["n"]), dtype=torch.int32, device="cuda"))
    return dict(case=c, w=w, d=torch.empty_like(w))


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "gemm":
        return apsp.tropical_gemm(state["out"], state["a"], state["b"])
    if kind == "pred":
        return apsp.apsp_predecessors(state["d"], state["w"], state["pred"])
    d = state["d"]
    d.copy_(state["w"])
    if kind == "fw":
        apsp.apsp_fw(d)
    elif kind == "rkleene":
        apsp.apsp_rkleene(d, cutoff=c["cutoff"])
    elif kind == "squaring":
        apsp.apsp_squaring(d)
    elif kind == "signed":
        apsp.apsp_fw_signed(d)
    elif kind == "cta":
        apsp.apsp_close_cta(d)
    else:
        apsp.apsp_batched_raw(d, state["offsets"], state["ns"], state["lds"], state["order"], c["count"],
                              state["ws"], ns_host=state["ns_host"])
    return d


def work(case):
    c = case
    if c["kind"] == "gemm":
        return {"bytes": 4 * (c["m"] * c["k"] + c["k"] * c["n"] + c["m"] * c["n"]),
                "flops": 2 * c["m"] * c["n"] * c["k"]}
    if c["kind"] == "batch":
        ns = [int(n) for n in _batch_layout(c)[0]]
        return {"bytes": 8 * sum(n ** 2 for n in ns), "flops": 2 * sum(n ** 3 for n in ns)}
    return {"bytes": (12 if c["kind"] == "pred" else 8) * c["n"] ** 2, "flops": 2 * c["n"] ** 3}


def _as64(w):
    w = w.to(torch.float64)
    return w.masked_fill_(w >= INF, math.inf)


def _back(d, dtype):
    return d.masked_fill_(d == math.inf, INF).to(torch.int64) if dtype == "i32" else d


def exact(case, seed):
    c = case
    if c["kind"] == "pred":
        return None  # indices
    if c["kind"] == "gemm":
        s = prepare(c, seed)
        a, b = _as64(s["a"]), _as64(s["b"])
        out = torch.full((c["m"], c["n"]), math.inf, dtype=torch.float64, device="cuda")
        for k in range(c["k"]):
            torch.minimum(out, a[:, k:k + 1] + b[k:k + 1], out=out)
        return _back(out, c["dtype"])
    if c["kind"] == "batch":
        pool, ns, (_, _, d_lds, d_offsets, _) = _batch_pool(c, seed)
        lds, offsets = d_lds.tolist(), d_offsets.tolist()
        out = pool.to(torch.float64 if c["dtype"] == "f32" else torch.int64)
        todo = {}
        for g, n in enumerate(ns.tolist()):  # graphs of about one size are closed together
            todo.setdefault((n + 63) // 64 * 64, []).append(g)
        for size, graphs in todo.items():
            for at in range(0, len(graphs), 128):
                some = graphs[at:at + 128]
                d = torch.full((len(some), size, size), math.inf, dtype=torch.float64, device="cuda")
                views = [pool[offsets[g]:offsets[g] + int(ns[g]) * lds[g]].view(int(ns[g]), lds[g]) for g in some]
                for x, g, v in zip(d, some, views):
                    x[:ns[g], :ns[g]] = _as64(v[:, :ns[g]])
                d.diagonal(dim1=1, dim2=2).zero_()
                d = _torch_closure(d, torch.float64)
                for x, g in zip(d, some):
                    n, o = int(ns[g]), offsets[g]
                    out[o:o + n * lds[g]].view(n, lds[g])[:, :n] = _back(x[:n, :n], c["dtype"])
        return out
    if c["n"] > 8192:
        return None
    return _back(_torch_closure(_as64(prepare(c, seed)["w"]), torch.float64), c["dtype"])
