"""The calls that a user of the memory store makes, as timed cases.

Every case goes through `MemStore`, the package's public interface.  Four
kinds of call:

    retrieve  a batch of queries against a store: scores, relation hops, top-k,
              pages; with or without hops, a namespace scope and time order
    ingest    a turn's new chunks: append, then the relation update that links
              them to the store (the graph is read back)
    forget    chunks deleted from the store and its graph (read back)
    manage    the Memory Manager after a batch of requests: relocation of
              co-retrieved chunks, then page compaction (the directory is read
              back)

Sizes are those of the repository's own workload configurations (`synth`)
and of sizes around and between them.  Stores are made on the GPU from the
seed: unit-length bf16 embeddings of a Gaussian mixture whose component
sizes fall with a Zipf law, or independent ones, and a relation graph that is
`popular` (targets by a power law, three quarters within the chunk's own
component: few chunks have very many in-links), `knn` (the nearest
neighbours within a component, as relation updates make them) or `uniform`.
"""
from __future__ import annotations

import ctypes
import math

import torch

from paper_2607_05708_gb300 import MemStore, load_library

DEV = "cuda"
ALPHA = 0.5           # weight of a hop, as in most of the workload configurations
SCALE = 10.0          # relation_scale: edge logit = SCALE * cosine


def _retrieve(name, n, dim, queries, hops, k, graph="popular", links=32, per_page=64,
              namespaces=0):
    return dict(name=name, kind="retrieve", n=n, dim=dim, queries=queries, hops=hops, k=k,
                graph=graph, links=links, per_page=per_page, namespaces=namespaces)


def _ingest(name, n, dim, new, m, links=32, rounds=16):
    return dict(name=name, kind="ingest", n=n, dim=dim, new=new, m=m, links=links, rounds=rounds,
                graph="popular", per_page=64, namespaces=0)


def listed():
    return [
        # a small agent's memory asked by a handful of users: the `tiny`
        # configuration, where latency and launches are all there is
        _retrieve("tiny_4q_1hop", 4096, 256, 4, 1, 8, graph="uniform", links=8, per_page=16),
        # one interactive query against a large shared memory
        _retrieve("large_1q_2hop", 1_048_576, 1024, 1, 2, 32),
        # a serving step's few concurrent requests on a mid-size memory of
        # ragged size
        _retrieve("mid_24q_2hop", 262_147, 768, 24, 2, 32),
        # the `gmm65k` configuration: a nearest-neighbour graph without heavy
        # in-degrees, one hop
        _retrieve("knn_64q_1hop", 65_536, 768, 64, 1, 16, graph="knn", links=16, per_page=32),
        # the `gmm1m` configuration: the full batch on the large memory
        _retrieve("large_256q_2hop", 1_048_576, 1024, 256, 2, 32),
        # tenants kept apart: every query in its namespace, results in time
        # order, an odd batch and store size
        _retrieve("scoped_100q_2hop", 500_009, 1024, 100, 2, 16, namespaces=64),
        # the Dense-only form of the paper's ablation: top 5, no hops
        _retrieve("dense_256q", 1_000_003, 1024, 256, 0, 5),
        # deep propagation with long result lists
        _retrieve("deep_200q_3hop", 262_144, 768, 200, 3, 64),
        # an agent's turn: a few dozen new chunks linked to a mid-size memory
        _ingest("turn_40new", 262_144, 1024, 40, 32, rounds=512),
        # a document import: the `update` configuration's 4096 new chunks
        _ingest("import_4096new", 1_048_576, 1024, 4096, 32, rounds=64),
        # a session's chunks forgotten
        dict(name="forget_200", kind="forget", n=524_288, dim=256, ids=200, links=32,
             graph="popular", per_page=64, namespaces=0),
        # the Memory Manager behind a batch of 256 top-5 requests on a large
        # directory
        dict(name="manage_256req", kind="manage", n=1_048_576, dim=64, requests=256, top=5,
             per_page=64, namespaces=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["retrieve"] * 6 + ["ingest"] * 2 + ["forget", "manage"])
    dim = rng.choice([64, 128, 192, 256, 384, 512, 768, 1024])
    if kind == "retrieve":
        while True:
            graph = rng.choice(["popular", "popular", "knn", "uniform"])
            # the nearest-neighbour and uniform graphs up to the size of the
            # configuration that has them
            n = _log_int(rng, 2_000, 1_048_576 if graph == "popular" else 65_536)
            queries = _log_int(rng, 1, 256)
            hops = rng.choice([0, 1, 2, 2, 2, 3])
            links = rng.choice([8, 16, 32])
            if graph == "knn":
                n = max(16, n // 128) * 128
            # no more edges to gather for than the deepest listed case, and
            # no more dots than the largest
            if n * links * queries * hops <= 262_144 * 32 * 200 * 3 and \
                    n * dim * queries <= 1_048_576 * 1024 * 256:
                break
        c = _retrieve("", n, dim, queries, hops, _log_int(rng, 1, 64), graph, links,
                      rng.choice([16, 32, 64]), rng.choice([0, 0, 0, 8, 64]))
    elif kind == "ingest":
        n = _log_int(rng, 8_192, 524_288)
        new = _log_int(rng, 1, 4096)
        c = _ingest("", n, dim, new, _log_int(rng, 1, 64), rng.choice([8, 16, 32]),
                    512 if new < 256 else 64)
    elif kind == "forget":
        c = dict(kind="forget", n=_log_int(rng, 8_192, 524_288), dim=dim,
                 ids=_log_int(rng, 1, 256), links=rng.choice([8, 16, 32]), graph="popular",
                 per_page=64, namespaces=0)
    else:
        c = dict(kind="manage", n=_log_int(rng, 8_192, 1_048_576), dim=64,
                 requests=_log_int(rng, 1, 256), top=rng.choice([3, 5, 8, 16]),
                 per_page=rng.choice([16, 64]), namespaces=rng.choice([1, 4, 64]))
    c.pop("name", None)
    return c


# --------------------------------------------------------------------------- inputs
def _components(n):
    return max(2, n // 256)


def _unit_bf16(x):
    return (x / x.norm(dim=1, keepdim=True)).to(torch.bfloat16)


def _mixture(gen, centers, comp, sigma):
    out = torch.empty((comp.numel(), centers.shape[1]), dtype=torch.bfloat16, device=DEV)
    for r0 in range(0, comp.numel(), 131_072):
        c = comp[r0:r0 + 131_072]
        x = torch.randn((c.numel(), centers.shape[1]), generator=gen, device=DEV)
        out[r0:r0 + 131_072] = _unit_bf16(x.mul_(sigma).add_(centers[c]))
    return out


def _first_distinct(t, rows, n, links):
    """The first `links` distinct targets of each row of draws `t` (the row's
    own chunk left out; the IDs after it where the draws repeat too often),
    ascending."""
    fill = (rows[:, None] + 1 + torch.arange(links, device=DEV)) % n
    srt, when = torch.sort(torch.cat([t, fill], 1), dim=1, stable=True)
    new = srt != rows[:, None]
    new[:, 1:] &= srt[:, 1:] != srt[:, :-1]
    last = torch.where(new, when, 4 * links).sort(dim=1).values[:, links - 1:links]
    return srt[new & (when <= last)].view(-1, links)


def _popular_graph(gen, n, links, comp, n_comp):
    """`links` distinct targets per chunk in proportion to a popularity
    rank^-1.1, three quarters of the draws within the chunk's component;
    logit 10 inside a component, 0 across, plus ln U."""
    pop = (torch.randperm(n, generator=gen, device=DEV) + 1).double().pow(-1.1)
    cs_all = pop.cumsum(0)
    members = torch.argsort(comp, stable=True)
    cs_in = pop[members].cumsum(0)
    bounds = torch.searchsorted(comp[members], torch.arange(n_comp + 1, device=DEV))
    lo = torch.cat([cs_in.new_zeros(1), cs_in])[bounds[:-1]]
    hi = torch.cat([cs_in.new_zeros(1), cs_in])[bounds[1:]]
    cols, affs = [], []
    for r0 in range(0, n, 131_072):
        rows = torch.arange(r0, min(n, r0 + 131_072), device=DEV)
        c = comp[rows]
        shape = (rows.numel(), 2 * links)
        u = torch.rand(shape, generator=gen, device=DEV, dtype=torch.float64)
        inside = torch.rand(shape, generator=gen, device=DEV) < 0.75
        at = torch.searchsorted(cs_in, lo[c][:, None] + u * (hi - lo)[c][:, None], right=True)
        at = torch.minimum(torch.maximum(at, bounds[c][:, None]), (bounds[c + 1] - 1)[:, None])
        t_all = torch.searchsorted(cs_all, u * cs_all[-1], right=True).clamp_(max=n - 1)
        t = _first_distinct(torch.where(inside, members[at], t_all), rows, n, links)
        jit = torch.log(1.0 - torch.rand(t.shape, generator=gen, device=DEV))
        cols.append(t.view(-1).int())
        affs.append((10.0 * (comp[t] == c[:, None]) + jit).view(-1))
    return (torch.arange(n + 1, device=DEV) * links, torch.cat(cols), torch.cat(affs))


def _uniform_graph(gen, n, links):
    t = torch.randint(0, n, (n, 2 * links), generator=gen, device=DEV)
    t = _first_distinct(t, torch.arange(n, device=DEV), n, links).view(-1).int()
    aff = torch.log(1.0 - torch.rand(t.shape, generator=gen, device=DEV))
    return torch.arange(n + 1, device=DEV) * links, t, aff


def _knn_graph(emb, comp, links):
    """The `links` nearest chunks of the same component (components of 128)."""
    n = emb.shape[0]
    members = torch.argsort(comp, stable=True).view(-1, 128)
    x = emb[members].float()
    g = torch.bmm(x, x.transpose(1, 2))
    g.diagonal(dim1=1, dim2=2).fill_(-math.inf)
    cos, at = g.topk(links, dim=2)
    t = torch.gather(members[:, None, :].expand(-1, 128, -1), 2, at)
    t, order = t.sort(dim=2)
    cos = cos.gather(2, order)
    col = torch.empty((n, links), dtype=torch.int64, device=DEV)
    aff = torch.empty((n, links), device=DEV)
    col[members.view(-1)] = t.view(n, links)
    aff[members.view(-1)] = SCALE * cos.view(n, links)
    return (torch.arange(n + 1, device=DEV) * links, col.view(-1).int(), aff.view(-1))


def _inputs(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(1_000_003 * (seed % 1_000_000_007) + 17)
    n, dim, kind = case["n"], case["dim"], case["kind"]
    x = {}
    uniform = case.get("graph") == "uniform"
    n_comp = n // 128 if case.get("graph") == "knn" else _components(n)
    centers = torch.randn((n_comp, dim), generator=gen, device=DEV)
    centers /= centers.norm(dim=1, keepdim=True)
    if case.get("graph") == "knn":
        comp = torch.arange(n, device=DEV) // 128
    else:
        # Zipf(1.1) sizes: the inverse of the cumulated weights
        cdf = torch.arange(1, n_comp + 1, device=DEV).double().pow(-1.1).cumsum(0)
        comp = torch.searchsorted(cdf / cdf[-1], (torch.arange(n, device=DEV) + 0.5) / n)
        comp = comp.clamp_(max=n_comp - 1)
    comp = comp[torch.randperm(n, generator=gen, device=DEV)]
    if uniform:
        x["emb"] = _unit_bf16(torch.randn((n, dim), generator=gen, device=DEV))
    else:
        x["emb"] = _mixture(gen, centers, comp, 0.3 / math.sqrt(dim))
    # chunks of a component packed on pages together
    pos = torch.empty(n, dtype=torch.int64, device=DEV)
    pos[torch.argsort(comp, stable=True)] = torch.arange(n, device=DEV)
    x["page_of"] = (pos // case["per_page"]).int()
    if kind != "manage":
        if uniform:
            x["row_ptr"], x["col"], x["aff"] = _uniform_graph(gen, n, case["links"])
        elif case["graph"] == "knn":
            x["row_ptr"], x["col"], x["aff"] = _knn_graph(x["emb"], comp, case["links"])
        else:
            x["row_ptr"], x["col"], x["aff"] = _popular_graph(gen, n, case["links"], comp, n_comp)
    if case["namespaces"]:
        x["ns"] = (comp % case["namespaces"]).int()
    if kind == "retrieve":
        b = case["queries"]
        if uniform:
            x["q"] = _unit_bf16(torch.randn((b, dim), generator=gen, device=DEV))
        else:
            qc = torch.randint(0, n_comp, (b,), generator=gen, device=DEV)
            x["q"] = _mixture(gen, centers, qc, 0.1 / math.sqrt(dim))
        if case["namespaces"]:
            x["q_ns"] = torch.randint(0, case["namespaces"], (b,), generator=gen, device=DEV).int()
    elif kind == "ingest":
        nc = comp[torch.randint(0, n, (case["rounds"] * case["new"],), generator=gen, device=DEV)]
        x["new"] = _mixture(gen, centers, nc, 0.3 / math.sqrt(dim))
    elif kind == "forget":
        x["gone"] = torch.randperm(n, generator=gen, device=DEV)[:n // 4]
    elif kind == "manage":
        # requests about recurring topics: a topic's chunks are mostly the
        # same ones each time
        top, topics = case["top"], max(64, n // 256)
        about = torch.randint(0, n, (topics, top + 2), generator=gen, device=DEV)
        w = torch.arange(1, topics + 1, device=DEV).double().pow(-1.1)
        pick = torch.multinomial(w, 64 * case["requests"], replacement=True, generator=gen)
        sets = about[pick]
        skip = torch.rand(sets.shape, generator=gen, device=DEV)
        skip[:, :top] *= 0.6
        sets = sets.gather(1, skip.argsort(dim=1)[:, :top])
        x["requests"] = sets.view(64, case["requests"], top).contiguous()
    return x


def _bits(t):
    return t.view(torch.int16)


def _store(case, x):
    st = MemStore(case["dim"], case["n"] + case.get("rounds", 0) * case.get("new", 0),
                  chunks_per_page=case["per_page"], relation_scale=SCALE)
    st.append_chunks(_bits(x["emb"]), x["page_of"], x.get("row_ptr"), x.get("col"), x.get("aff"))
    if "ns" in x:
        st.set_namespace(0, x["ns"])
    return st


def prepare(case, seed):
    x = _inputs(case, seed)
    state = {"case": case, "store": _store(case, x), "at": 0}
    if case["kind"] == "retrieve":
        state["q"], state["q_ns"] = _bits(x["q"]), x.get("q_ns")
    else:
        state["x"] = x
    return state


# --------------------------------------------------------------------------- one pass
def _export(st, n, room):
    """The graph read back into buffers with room for `room` edges (zeros past
    the graph's own), through the C interface."""
    lib, stream = load_library(), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    out = {"row_ptr": torch.empty(n + 1, dtype=torch.int64, device=DEV),
           "col": torch.empty(room, dtype=torch.int32, device=DEV),
           "aff": torch.empty(room, device=DEV), "w": torch.empty(room, device=DEV)}
    p = {k: ctypes.c_void_p(t.data_ptr()) for k, t in out.items()}
    rows, nnz = ctypes.c_int64(), ctypes.c_int64()
    if lib.akashic_mem_export_csr(st._h, ctypes.byref(rows), ctypes.byref(nnz), p["row_ptr"],
                                  p["col"], p["aff"], p["w"], stream):
        raise RuntimeError(lib.akashic_mem_last_error().decode())
    for k in ("col", "aff", "w"):
        out[k][nnz.value:].zero_()
    return out


def run(state):
    case, st = state["case"], state["store"]
    if case["kind"] == "retrieve":
        scoped = bool(case["namespaces"])
        ids, scores, pages, n_pages = st.retrieve(state["q"], case["k"], ALPHA, case["hops"],
                                                  q_ns=state["q_ns"], sort_by_time=scoped)
        return {"ids": ids, "scores": scores, "pages": pages, "n_pages": n_pages}
    x, i = state["x"], state["at"]
    state["at"] = i + 1
    if case["kind"] == "ingest":
        n, at = case["new"], i % case["rounds"]
        if i and at == 0:                # the store is full: the memory starts over
            st.close()
            st = state["store"] = _store(case, x)
        first = st.append_chunks(_bits(x["new"][at * n:(at + 1) * n]))
        st.update_relations(first, n, case["m"], True)
        row_ptr, col, aff, w = st.export_csr()
        new = -n * case["m"]             # the new rows are the last ones
        return {"row_ptr": row_ptr, "col": col, "aff": aff, "w": w, "aff_new": aff[new:],
                "w_new": w[new:]}
    if case["kind"] == "forget":
        n, rounds = case["ids"], x["gone"].numel() // case["ids"]
        at = i % rounds
        if i and at == 0:                # a quarter is gone: the memory starts over
            st.close()
            st = state["store"] = _store(case, x)
        st.delete(x["gone"][at * n:(at + 1) * n])
        return _export(st, case["n"], case["n"] * case["links"])
    st.relocate(x["requests"][i % 64], 0.7)
    released = st.compact_pages(0.75, 0.7)
    return {"released": released, "pages": st.export_pages(), **st.page_stats()}


# --------------------------------------------------------------------------- what it takes
def work(case):
    n, d, kind = case["n"], case["dim"], case["kind"]
    if kind == "manage":
        # the directory read back, the requests, their statistics
        return {"bytes": 8 * n + case["requests"] * case["top"] * 8.0, "flops": 0}
    nnz = n * case["links"]
    if kind == "retrieve":
        b = case["queries"]
        graph = 8 * (n + 1) + 8 * nnz if case["hops"] else 0      # (source, weight) once
        out = b * case["k"] * 16 + b * 4
        return {"bytes": 2 * n * d + 2 * b * d + graph + 4 * n * bool(case["namespaces"]) + out,
                "flops": 2.0 * n * d * b}
    if kind == "ingest":
        new = case["new"]
        # the store's rows read once, the new ones read and written, the graph
        # read back (copied: read and written), its new edges written both ways
        edges = nnz + 2 * new * case["m"]
        return {"bytes": 2 * n * d + 4 * new * d + 24 * edges + 16 * n + 48 * new * case["m"],
                "flops": 2.0 * new * n * d}
    # both edge lists compacted (12 bytes an edge read and written each), then
    # read back
    return {"bytes": 3 * 24 * nnz + 3 * 16 * n, "flops": 0}


# What a correct implementation of the same precision may differ by (about
# four times what was seen against 64 bits).
def tolerance(case):
    if case["kind"] == "manage":
        return "exact"
    if case["kind"] == "retrieve":
        # fp32 scores over a sum of n of them; IDs (and the pages with them)
        # may swap where two scores are equal in 32 bits
        # (6e-6 and 1.1e-5 seen at worst, where the terms of the hops are
        # 16-bit pairs; 0.5% of the IDs without hops)
        return {"rel": 2.5e-5, "max": 5e-5, "differ": 0.01}
    if case["kind"] == "ingest":
        # logits are 10 * a 32-bit dot, weights their softmax: 1.5e-6 apart,
        # 4e-4 with the few neighbours of equal cosine that swap in an import
        return {"rel": 2e-3, "max": 0.2, "differ": 1e-3}
    # weights only: 6e-8 and 1.3e-6 seen
    return {"rel": 3e-7, "max": 5e-6, "differ": 0.0}


# --------------------------------------------------------------------------- 64 bits
def _softmax64(row_ptr, aff):
    n = row_ptr.numel() - 1
    rows = torch.repeat_interleave(torch.arange(n, device=DEV), row_ptr[1:] - row_ptr[:-1])
    a = aff.double()
    top = torch.full((n,), -math.inf, dtype=torch.float64, device=DEV)
    top.scatter_reduce_(0, rows, a, "amax")
    e = (a - top[rows]).exp()
    z = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, rows, e)
    return e / z[rows]


def _exact_retrieve(case, x):
    n, d, b, k = case["n"], case["dim"], case["queries"], case["k"]
    q = x["q"].double()
    tau = 1.0 / math.sqrt(d)
    z = torch.empty((n, b), dtype=torch.float64, device=DEV)
    for r0 in range(0, n, 65_536):
        z[r0:r0 + 65_536] = x["emb"][r0:r0 + 65_536].double() @ q.t()
    u = z.mul_(tau)
    u = u.sub_(u.max(dim=0).values).exp_()
    s = u
    if case["hops"]:
        w = _softmax64(x["row_ptr"], x["aff"])
        rows = torch.repeat_interleave(torch.arange(n, device=DEV),
                                       x["row_ptr"][1:] - x["row_ptr"][:-1])
        order = torch.argsort(x["col"], stable=True)      # the transpose: in-edges
        in_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
        in_ptr[1:] = torch.bincount(x["col"], minlength=n).cumsum(0)
        r_t = torch.sparse_csr_tensor(in_ptr, rows[order], w[order], size=(n, n))
        for _ in range(case["hops"]):
            s = u + ALPHA * (r_t @ s)
    s = s / u.sum(dim=0)
    if case["namespaces"]:
        s = torch.where(x["ns"][:, None] == x["q_ns"][None, :], s, -1.0)
    top, ids = s.t().contiguous().topk(k, dim=1)
    pad = top < 0
    if case["namespaces"]:                                # results in time order
        ids = torch.where(pad, n, ids)
        ids, order = ids.sort(dim=1)
        top, pad = top.gather(1, order), pad.gather(1, order)
        ids = torch.where(pad, 0, ids)
    pages = torch.where(pad, -1, x["page_of"][ids])
    srt = pages.sort(dim=1).values
    n_pages = (srt[:, :1] >= 0).sum(1) + ((srt[:, 1:] != srt[:, :-1]) & (srt[:, 1:] >= 0)).sum(1)
    return {"ids": torch.where(pad, -1, ids), "scores": torch.where(pad, 0.0, top),
            "pages": pages.int(), "n_pages": n_pages.int()}


def _exact_ingest(case, x):
    n, m, new = case["n"], case["m"], case["new"]
    e = x["new"][:new].double()
    best, ids = torch.full((new, 1), -9.0, dtype=torch.float64, device=DEV), None
    for r0 in range(0, n, 65_536):
        dots = e @ x["emb"][r0:r0 + 65_536].double().t()
        v, at = dots.topk(min(m, dots.shape[1]), dim=1)
        best = v if ids is None else torch.cat([best, v], 1)
        ids = at + r0 if ids is None else torch.cat([ids, at + r0], 1)
        best, sel = best.topk(min(m, best.shape[1]), dim=1)
        ids = ids.gather(1, sel)
    ids, order = ids.sort(dim=1)
    aff = SCALE * best.gather(1, order)
    w = torch.softmax(aff, dim=1)
    # the whole lists are left out: one swap of two neighbours with equal
    # cosines would shift a part of them by an edge
    return {"row_ptr": None, "col": None, "aff": None, "w": None, "aff_new": aff.view(-1),
            "w_new": w.view(-1)}


def _exact_forget(case, x):
    n = case["n"]
    dead = torch.zeros(n, dtype=torch.bool, device=DEV)
    dead[x["gone"][:case["ids"]]] = True
    rows = torch.repeat_interleave(torch.arange(n, device=DEV),
                                   x["row_ptr"][1:] - x["row_ptr"][:-1])
    keep = ~dead[rows] & ~dead[x["col"].long()]
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    row_ptr[1:] = torch.bincount(rows[keep], minlength=n).cumsum(0)
    aff, pad = x["aff"][keep], (0, x["col"].numel() - int(keep.sum()))
    return {"row_ptr": row_ptr, "col": torch.nn.functional.pad(x["col"][keep], pad),
            "aff": torch.nn.functional.pad(aff.double(), pad),
            "w": torch.nn.functional.pad(_softmax64(row_ptr, aff), pad)}


def exact(case, seed):
    if case["kind"] == "manage":
        return None                                       # whole numbers only
    x = _inputs(case, seed)
    return {"retrieve": _exact_retrieve, "ingest": _exact_ingest,
            "forget": _exact_forget}[case["kind"]](case, x)
